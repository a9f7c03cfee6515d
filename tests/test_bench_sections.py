"""bench.py's sections: every result goes to stderr when it ends, an error is the
section's result, and a section that does not end within its limit leaves the line
with what was measured before it."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import time, bench
sec = bench.Sections(1.0)
sec.line = {"metric": "m", "value": 3.0}
sec.line["first"] = sec.run("first", lambda: {"x": 1})
sec.line["bad"] = sec.run("bad", lambda: 1 / 0)
sec.run("stuck", lambda: time.sleep(60))
print("not reached")
"""


def test_sections_report_and_end():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=50)
    assert r.returncode == 0, r.stderr
    out = r.stdout.strip().splitlines()
    assert len(out) == 1
    line = json.loads(out[0])
    assert line["value"] == 3.0 and line["first"] == {"x": 1} and "ZeroDivisionError" in line["bad"]["error"]
    assert line["unfinished"] == "stuck"
    assert "first {" in r.stderr and "stuck: time limit" in r.stderr
