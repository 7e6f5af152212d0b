"""The timeline's report on stamps made by hand: which points it names, when a kernel ends, in which order kernels ran."""
import numpy as np

from paper_2402_13720_b200 import trace


def _stamps():
    return np.zeros((8, 160, 16), dtype=np.int64), np.zeros((512, 8), dtype=np.int64)


def _line(lines, name):
    return next(ln for ln in lines if name in ln)


def test_wide_blocks_end_with_the_fix_up():
    g, a = _stamps()
    g[1, :3, 1] = 5000
    g[1, :3, 4] = 7000
    g[1, :3, 5] = 8000
    g[1, :2, 7] = 9500
    lines = trace.report(g, a, False)
    assert "max    2.0" in _line(lines, "last accumulator complete")
    assert lines[-1].split() == ["o-proj", "0.0", "4.5", "4.5"]
    assert not any("attention" in ln for ln in lines)


def test_a_single_row_ends_with_its_outputs():
    """gemm_rows_kernel stamps some of the same slots with other meanings, and others not at all."""
    g, a = _stamps()
    g[2, :148, 1] = 20000
    g[2, 140:148, 1] = 16000                     # CTAs with nothing to do in the GEMM before
    g[2, :148, 4] = 21200
    g[2, :148, 2] = 21500
    g[2, :148, 3] = 26000
    g[2, :148, 5] = 26300
    g[2, :148, 10] = 27100
    a[:8, 0] = 12000
    a[:8, 2] = 13000                             # waits are over ahead of the GEMM
    a[:8, 5] = 16400
    a[8, 0] = 12000                              # a CTA without keys stamps its entry only
    lines = trace.report(g, a, True)
    assert "med   -1.2" in _line(lines, "activations asked for") and "max    5.9" in _line(lines, "outputs written")
    assert not any("accumulator" in ln or "fix-up" in ln for ln in lines)
    assert [ln.split() for ln in lines[-2:]] == [["attention", "0.0", "3.4", "3.4"], ["gate,up", "8.2", "14.1", "5.9"]]


def test_nothing_stamped():
    assert len(trace.report(*_stamps(), False)) == 1
