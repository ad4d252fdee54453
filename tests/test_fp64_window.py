"""The window in which an FP64 context's walks take Eq. 5 again in FP64, with the kernels'
float arithmetic emulated in numpy: every case whose FP32 decision differs from the FP64 one
lies inside wa d2 + wb (wa = 4e-6 + 16 b / side, wb = b side / 64 + 1e-37, b = 5e-7 X, X the
target's largest coordinate) in any unit of length, and in every unit that window holds the
same small share of the cases."""
import numpy as np
import pytest

from test_fp32_window import _cases, _f32, _fma32


def _decide(x, c, rc2, side):
    """FP32 decisions and whether each lies inside the window."""
    with np.errstate(over="ignore", invalid="ignore"):
        xh, ch = _f32(x), _f32(c)
        R = _f32(xh - ch)
        d2 = _fma32(R[:, 0], R[:, 0], _fma32(R[:, 1], R[:, 1], _f32(R[:, 2] * R[:, 2])))
        dm = _f32(d2 - np.minimum(_f32(rc2), np.finfo(np.float32).max))
        b = _f32(_f32(5e-7) * np.abs(xh).max(axis=1))
        wa = _fma32(b, _f32(16.0 / side), _f32(4e-6))
        wb = _fma32(b, _f32(_f32(side) / 64.0), _f32(1e-37))
        win = _fma32(wa, d2, wb)
        return dm > 0, ~(np.abs(dm) > win)


@pytest.mark.parametrize("unit", [-130, -62, -40, -20, 0, 20, 40, 62, 64, 130])
def test_decisions_and_share(unit):
    f = 2.0 ** unit
    for scale, seed in ((1.0, 1), (40.0, 2), (1000.0, 3)):
        for rel in (1e-4, 3e-7):
            x, c, rc2 = _cases(100000, scale, seed, rel=rel)
            exact = ((x - c) ** 2).sum(axis=1) > rc2
            got, inside = _decide(x * f, c * f, rc2 * f * f, 2 * scale * f)
            assert np.array_equal(got[~inside], exact[~inside])
            if abs(unit) <= 40:
                assert inside.mean() <= _decide(x, c, rc2, 2 * scale)[1].mean() + 1e-3
