"""The benchmark's result line: one short JSON line on stdout with the headline,
whatever the other arms measured; their tables on stderr."""
import json

import bench


def test_the_headline_is_short_and_alone_on_stdout(capsys):
    table = [[63.203 + i for i in range(12)] for _ in range(300)]
    line = {"metric": bench.METRIC, "value": 6.95e8, "unit": "moves/s", "config": bench.bench_config(bench.parse_args([])),
            "clocks": {"sm_mhz": 2070.0, "reasons": []}, "gpu_launches": 40}
    bench.print_line({**line, **{k: {"table": table} for k in bench.ARMS}})
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 1500
    assert json.loads(out) == line
    assert set(json.loads(err)["arms"]) == set(bench.ARMS)
    bench.print_line({**line, **{k: None for k in bench.ARMS}})
    out, err = capsys.readouterr()
    assert json.loads(out) == line and err == ""


def test_every_arm_of_the_line_is_known():
    src = open(bench.__file__).read()
    body = src[src.index('"cpu_baseline": cpu,'):src.index("print_line(line)\n    g.close()")]
    assert [k for k in bench.ARMS if '"%s"' % k not in body] == []
