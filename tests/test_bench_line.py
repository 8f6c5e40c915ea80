"""bench.py's printed line holds the headline numbers in less than 3000 characters, whatever the full
record grows to; the record goes to a file."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench


def _record():
    number = 0.12345678901234567
    text = "x" * 120
    line = {k: number for k in bench.HEADLINE}
    line["config"] = {"k%02d" % i: number for i in range(13)}
    line["roofline"] = {"kernel": text, "bound": "alu", **{"k%d" % i: number for i in range(8)}}
    line["cpu_baseline"] = {"sample": text, "cpu_model": "Neoverse-V2", **{"k%d" % i: number for i in range(4)}}
    for k, notes in bench.NOTES.items():
        line[k].update((q, text * 5) for q in notes)
    line["e2e"] = {"value": number, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 9, "d2h_bytes_per_step": 10 ** 9}
    line["clocks"] = {"sm_mhz": number, "sm_max_mhz": number, "reasons": [text]}
    for i in range(200):
        line["secondary_%d" % i] = {"note": text}
    return line


def test_printed_line(capsys, tmp_path):
    line, path = _record(), tmp_path / "d.json"
    bench.emit(line, str(path))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 3000
    got = json.loads(out)
    assert list(got) == bench.HEADLINE
    for k, v in got.items():
        drop = bench.NOTES.get(k, ())
        assert v == ({q: x for q, x in line[k].items() if q not in drop} if drop else line[k])
    assert json.loads(path.read_text()) == line


def test_contract_keys_are_in_the_line():
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "clocks", "gpu_launches"):
        assert k in bench.HEADLINE


def test_details_are_optional(capsys, tmp_path):
    line = _record()
    bench.emit(line, "")
    bench.emit(line, str(tmp_path / "missing" / "d.json"))
    got = capsys.readouterr()
    assert got.out.count("\n") == 2 and "details not written" in got.err
