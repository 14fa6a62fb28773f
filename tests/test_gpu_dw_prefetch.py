"""The dW GEMM's L2 prefetch of the next tile's dW lines (few masked rows, dW larger than L2).

The smallest dW that prefetches, with a ragged last vocabulary block and a
32-column last hidden-size tile, the same just below the size line, a hidden
size whose rows do not start on 128-byte lines (no prefetch), and K on both
sides of the 3,072-row line: l, dX and dW against the fp64 oracle within the tolerances of
the parity tests (l 1e-3 relative, gradients 2e-2 normwise).
"""
import numpy as np
import pytest

from synth import Workload, make_inputs
from tests.harness import ensure_built, gpu_run, normwise, oracle_run, rel_ell_err, to64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


@pytest.mark.parametrize("R,H,V,pair", [
    (20, 2080, 16201, False),    # 2^27 bytes of dW; V % 256 = 73
    (20, 2080, 16000, False),    # below 2^27 bytes
    (20, 2056, 16400, False),    # H % 32 != 0
    (20, 2080, 16201, True),     # K over a pending sample's rows too
    (1030, 1024, 32800, False),  # 467 and 1,616 rows
    (1030, 1024, 32800, True),   # K = 2,128 rows
    (1600, 1024, 32800, True),   # K over 3,072 rows: past the line
])
def test_prefetching_dw_matches_the_oracle(R, H, V, pair):
    wl = Workload("dw_prefetch", B=2, P=3, R=R, H=H, V=V, n_t=2, G=2, t_mode=1, seed=21,
                  targets="zipf", advantages="normal", eps_std=0.1)
    inp = make_inputs(wl)
    o = oracle_run(wl, inp)
    g = gpu_run(wl, {k: (v.cuda() if v is not None else None) for k, v in inp.items()},
                pair_dw=pair)
    assert np.array_equal(g["masks"].cpu().numpy(), o["masks"])
    assert rel_ell_err(to64(g["ell"]), o["ell"]).max() <= 1e-3
    assert np.linalg.norm(o["dW"]) > 0
    assert normwise(to64(g["dW"]), o["dW"]) <= 2e-2
    assert normwise(to64(g["dX"]), o["dX"]) <= 2e-2
