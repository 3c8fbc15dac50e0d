"""The plan tuner's record: what a choice is reused for, in the process and through MM_TUNE_CACHE."""
import json
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCAN = dict(nx=8, ny=8, n_det=2, n_t=4 * 4571, n_int=4, half_bw=37, f_knee=1.0, seed=4)


def child(cache, body):
    """Runs `body` in a fresh process (an empty record) with the given cache file; returns what it prints as JSON."""
    code = ("import sys, json, numpy as np; sys.path.insert(0, 'tests')\nimport synth\n"
            "import paper_1801_08937_gb300.mapmaker as MM\n" + textwrap.dedent(body))
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, MM_TUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


PRODUCT = f"""
    scan = synth.make_scan(**{SCAN!r})
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.setup_scan(scan)
    c.apply_A(np.zeros((1, scan.n_pix, 3)))
    print(json.dumps([c.get_option("plan_whole"), c.get_option("plan_fft_len")]))
"""


def test_lines_of_another_set_of_plans_are_passed_over(tmp_path):
    cache = tmp_path / "tune"
    child(cache, PRODUCT)
    lines = cache.read_text().splitlines()
    assert len(lines) == 1
    entry = json.loads(lines[0])
    forced = dict(entry, variant=2, L=256, whole=0, V=256 - 2 * 37)

    def lines_after(d):
        cache.write_text(json.dumps(d) + "\n")
        plan = child(cache, PRODUCT)
        return plan, len(cache.read_text().splitlines())

    assert lines_after(forced) == ([0.0, 256.0], 1)   # this build's own lines are used
    # others, and those from before lines carried a version: tuned again, recorded beside the old line
    assert lines_after(dict(forced, v=entry["v"] - 1))[1] == 2
    assert lines_after({k: v for k, v in forced.items() if k != "v"})[1] == 2
