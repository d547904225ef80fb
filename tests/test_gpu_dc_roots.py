"""The divide and conquer's reciprocals and roots on the GPU against correctly rounded
ones, within the bounds that their series and roundings give."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

dp = ctypes.POINTER(ctypes.c_double)


def test_errors_within_their_bounds():
    rng = np.random.default_rng(3)
    x = np.concatenate([2.0 ** rng.uniform(-1000, 1000, 40000),       # beyond float32: the library's functions
                        2.0 ** rng.uniform(-126, 126, 200000), rng.uniform(0.5, 2.0, 200000),
                        1.0 + 2.0 ** -52 * np.arange(64), 2.0 - 2.0 ** -52 * np.arange(1, 65),
                        [1e-37, 1e37, 1e-36, 2.0 ** -126, 2.0 ** 127, 2.0 ** -1022, 1.7e308]])
    out = [np.full_like(x, np.nan) for _ in range(3)]
    st = pkg.load().dsrg_fno_debug_dc_roots(len(x), x.ctypes.data_as(dp), *[o.ctypes.data_as(dp) for o in out])
    assert st == 0
    xl = x.astype(np.longdouble)
    want = [1 / xl, 1 / np.sqrt(xl), np.sqrt(xl)]
    # one rounding; that of x r in e (half of it) and the last one; those and the product's;
    # a result below 2^-1022 (1 / 1.7e308) is rounded to 2^-1074
    for got, ref, units in zip(out, want, (1.0, 1.5, 2.5)):
        assert np.all(np.abs(got - ref) <= (units + 0.01) * 2.0 ** -53 * ref + np.longdouble(2.0) ** -1075)
