"""dX under every kind of plan: 256- and 512-wide tiles, split and unsplit, one or
several vocabulary chunks, ragged hidden sizes and last row blocks. dX against
the fp64 oracle (2e-2 normwise, the parity tests' tolerance), rows no sample
masked exactly zero, and the same bits from a second run.
"""
import numpy as np
import pytest

from synth import Workload, make_inputs
from tests.harness import ensure_built, gpu_run, normwise, oracle_run, to64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,R,H,V,chunk", [
    (1, 300, 1032, 900, 0),      # 256-wide, few splits
    (2, 700, 2712, 500, 0),      # 256-wide, unsplit
    (2, 700, 2712, 1300, 512),   # unsplit or split, added over three chunks
    (1, 40, 104, 9000, 0),       # one column block, 16 splits
    (1, 40, 808, 3000, 1024),    # split, three chunks
    (4, 600, 200, 3000, 0),      # many row blocks, one column block
    (3, 200, 4096, 700, 0),      # a full-width head, short K
    (3, 260, 2056, 6000, 0),     # a last column block of 8
])
def test_dx_plans_match_the_oracle(B, R, H, V, chunk):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    wl = Workload("dx_plan", B=B, P=1, R=R, H=H, V=V, n_t=2, G=1, t_mode=1, seed=17 + H + V,
                  targets="zipf", advantages="normal", eps_std=0.1)
    inp = make_inputs(wl)
    o = oracle_run(wl, inp)
    dev = {k: (v.cuda() if v is not None else None) for k, v in inp.items()}
    a, b = (gpu_run(wl, dev, vocab_chunk=chunk) for _ in range(2))
    got = to64(a["dX"])
    assert np.linalg.norm(o["dX"]) > 0
    assert normwise(got, o["dX"]) <= 2e-2
    assert not got[~o["masks"].any(axis=0).astype(bool)].any()
    assert torch.equal(a["dX"], b["dX"]) and torch.equal(a["dW"], b["dW"])
