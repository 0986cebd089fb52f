"""The fp32 expansion at the sizes where its thread mapping can go wrong: rows around the 16 of a CTA, retained lengths around the 32 a pass of
loads takes and beyond the 256 threads, block lengths around the 64-position chunks and off the 16-byte rows, both one-sided modes.
Bound: the fp32 regression bound of the parity tests (5e-6 of the largest output: fp32 sums of up to 1000 terms)."""
import pytest

from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("mode", ["kv", "k", "v"])
@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (1, 1, 1, 3, 1, 2, 900), (1, 5, 1, 8, 3, 0, 500), (4, 4, 1, 9, 1, 7, 600), (1, 17, 1, 11, 1, 3, 730), (2, 6, 2, 16, 2, 20, 200),
    (1, 3, 1, 27, 2, 5, 550), (2, 4, 2, 16, 1, 3, 750), (2, 4, 2, 16, 1, 3, 746),       # (the last two: m = 64 and 66)
])
def test_fp32_expansion(B, H_q, H_kv, grid, R, T, ratio, mode):
    if H_q // H_kv > 16:
        H_q = 16
    shape = wl.Shape("fp32-expand", 1, B, H_q, H_kv, 128, grid, R, T, 1, "f32", ratio)
    p = tl.make_problem(shape, 400 + grid, T=T, T_cap=T + 1, recipe="peaked")
    _, _, _, out = tl.gpu_run(shape, p, mode=mode)
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused", mode)[2], "f32", mode)


@pytest.mark.parametrize("grid,ratio,mode", [(43, 110, "kv"), (48, 580, "k"), (48, 570, "k"), (48, 570, "v")])
def test_most_retained_rows_that_fit(grid, ratio, mode):
    """A score and a weight row of 3280 and of 3296 entries together, all that a CTA's shared memory holds."""
    n = grid * grid
    m = (n * (1000 - ratio) + 999) // 1000
    pitch = lambda x: (x + 15) // 16 * 16
    assert pitch(n if mode == "v" else m) + pitch(n if mode == "k" else m) == (3280 if ratio == 580 else 3296)
    shape = wl.Shape("fp32-long", 1, 1, 2, 1, 128, grid, 1, 3, 1, "f32", ratio)
    p = tl.make_problem(shape, 500 + grid, T=3, T_cap=4, recipe="peaked")
    _, _, _, out = tl.gpu_run(shape, p, mode=mode)
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused", mode)[2], "f32", mode)
