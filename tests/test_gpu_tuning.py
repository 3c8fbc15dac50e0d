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


# 64 blocks have fewer CTAs than the device has SMs, 256 blocks more (one CTA a block is then usual)
@pytest.mark.parametrize("n_det", [8, 32])
def test_half_transform_is_part_of_what_a_choice_is_reused_for(n_det):
    """0 keeps half-length plans out, 2 takes blocks split over two CTAs, whatever was tuned before for the
    other values; native float64, all tuned in one process."""
    import numpy as np
    import synth
    scan = synth.make_scan(nx=16, ny=16, n_det=n_det, n_t=8 * 4096, n_int=8, half_bw=500, f_knee=1.0, seed=8)
    got = []
    for half in (0, 1, 2, 1, 0, 2):
        c = MM.Context(0, None, MM.MM_FP64)
        c.set_option("half_transform", half)
        c.setup_scan(scan)
        c.apply_A(np.zeros((1, scan.n_pix, 3)))
        got.append(c.get_option("plan_whole"))
        c.close()
    assert got[0] in (0, 1) and got[4] == got[0]
    assert got[2] == got[5] == 3
    assert got[3] == got[1]


def test_template_products_record_no_plan(tmp_path):
    """The template kernel is one for every plan: its times say nothing about an unfiltered scan of the same shape."""
    cache = tmp_path / "tune"
    body = f"""
        scan = synth.make_scan(**{dict(SCAN, half_bw=0, f_knee=0.0, hwp=False)!r})
        sub, az, bins = synth.make_templates(scan)
        c = MM.Context(0, None, MM.MM_FP32_MIXED)
        c.setup_scan(scan)
        x = np.random.default_rng(1).standard_normal((1, scan.n_pix, 3))
        for on in (True, False):
            if on: c.set_templates(1, sub, az, bins)
            else: c.set_templates()
            c.apply_A(x)
            c.rhs(np.zeros((1, scan.n_samples), dtype=np.float32))
            if on: assert not __import__("os").path.exists({str(cache)!r})
        print(json.dumps(c.get_option("plan_whole")))
    """
    child(cache, body)
    assert len(cache.read_text().splitlines()) == 2   # the unfiltered float32 and double-float products


@pytest.mark.parametrize("prec", [MM.MM_FP64, MM.MM_FP32_MIXED])
def test_a_batch_chooses_between_few_plans(prec):
    """The first batch on a scan of few blocks does not time every plan again: four at most, each with a
    one-CTA warm-up and up to three timed launches, and tables (up to seven kernels) for those that are new;
    the batch's product stays the single ones'."""
    import numpy as np
    import synth
    from helpers import assert_close
    scan = synth.make_scan(nx=16, ny=16, n_det=8, n_t=8 * 3001, n_int=8, half_bw=301, f_knee=1.0, seed=12)
    c = MM.Context(0, None, prec)
    c.setup_scan(scan)
    x = np.random.default_rng(2).standard_normal((16, scan.n_pix, 3))
    one = [c.apply_A(v[None])[0] for v in x]
    n0 = c.get_option("kernel_launches")
    y = c.apply_A(x)
    n1 = c.get_option("kernel_launches")
    c.apply_A(x)
    n2 = c.get_option("kernel_launches")
    assert (n1 - n0) - (n2 - n1) <= 4 * (1 + 3 + 7)
    for a, b in zip(y, one):
        assert_close(a, b, 1e-12 if prec == MM.MM_FP64 else 1e-5)
    c.close()
