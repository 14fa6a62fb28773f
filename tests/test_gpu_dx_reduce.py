"""The split reduction of dX over its row-wise and flat forms: hidden sizes on both
sides of the 2,048-column line, vector counts that are no multiple of a tile, a
few and thousands of masked rows. dX against the fp64 oracle (2e-2 normwise, the
parity tests' tolerance), and rows no sample masked exactly zero.
"""
import numpy as np
import pytest

from synth import Workload, make_inputs
from tests.harness import ensure_built, gpu_run, normwise, oracle_run, to64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [64, 200, 1000, 2048, 2056])
@pytest.mark.parametrize("B,R", [(1, 5), (2, 150), (3, 700)])
def test_dx_reduction_matches_the_oracle(B, R, H):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    wl = Workload("dx_reduce", B=B, P=1, R=R, H=H, V=900, n_t=2, G=1, t_mode=1, seed=31 + H,
                  targets="zipf", advantages="normal", eps_std=0.1)
    inp = make_inputs(wl)
    o = oracle_run(wl, inp)
    g = gpu_run(wl, {k: (v.cuda() if v is not None else None) for k, v in inp.items()})
    got = to64(g["dX"])
    assert np.linalg.norm(o["dX"]) > 0
    assert normwise(got, o["dX"]) <= 2e-2
    assert not got[~o["masks"].any(axis=0).astype(bool)].any()
