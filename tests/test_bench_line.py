"""The benchmark's result line stays short whatever the extra workloads report."""
import json

import bench


def test_extras_do_not_lengthen_the_result_line(capsys):
    line = {"metric": "MLUPS", "value": 1.0, "unit": "MLUPS", "config": {"workload": "800^3"}}
    extra = {"c_sweep": {f"C={c}": {"E": [1.0 / (k + 1) for k in range(600)]} for c in range(4)}}
    bench.print_result(line, extra)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and json.loads(out) == line
    assert err.count("\n") == 1 and json.loads(err) == {"extra": extra}
    bench.print_result(line, {})
    assert capsys.readouterr() == (out, "")
