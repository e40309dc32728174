"""What the benchmark prints: the headline alone on stdout, short enough to be read from the end of the output."""
import json

import bench


def test_headline_is_short_and_the_tables_are_apart(capsys):
    res = {"metric": "m", "value": 1.0, **{name: list(range(5000)) for name in bench.TABLES}}
    bench.print_result(res)
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": "m", "value": 1.0} and out.count("\n") == 1
    assert [list(json.loads(line)) for line in err.splitlines()] == [[name] for name in bench.TABLES]
