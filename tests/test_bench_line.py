"""The benchmark's stdout is its one line, short enough to be kept whole; the
other workloads' summaries go to stderr."""
import json

import bench


def test_details_stay_off_the_line(capsys):
    line = {"metric": bench.METRIC, "value": 5164.603912345678, "clocks": {"reasons": []},
            "config": {"global_batch": 16384, "seq_len": None}}
    details = {"workloads": {f"w{i}": {"us": i / 7, "list": [i / 3, True, None, "x"]} for i in range(400)}}
    bench.emit(line, details)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 400
    got = json.loads(out)
    assert got["value"] == 5164.604 and got["config"] == line["config"]
    back = json.loads(err)["details"]["workloads"]
    assert back["w10"]["us"] == float(f"{10 / 7:.7g}") and back["w10"]["list"][1:] == [True, None, "x"]
