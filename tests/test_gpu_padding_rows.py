"""Rows past the masked ones: what the workspace holds there never reaches a result.

The GEMMs neither load A tiles nor write dZ, logits or split partials for CTAs
and warps whose rows are all unmasked (dZ keeps zeros up to the dW GEMM's next
64-row K block). A workspace full of NaN patterns must give the bits a zeroed
one gives, and the fp64 oracle's values (l 1e-3 relative, gradients 2e-2
normwise), at masked-row counts around 32, 64, 128 and 256.
"""
import numpy as np
import pytest

from synth import Workload, make_inputs
from tests.harness import ensure_built, normwise, oracle_run, rel_ell_err, to64

pytestmark = pytest.mark.gpu

# (B, R): masked rows per sample 1 .. 300 (stratified t: the last sample masks nearly all)
SIZES = [(1, 33), (1, 66), (1, 131), (2, 100), (1, 260), (3, 100)]


@pytest.mark.parametrize("B,R", SIZES)
@pytest.mark.parametrize("keep,pair", [(False, False), (False, True), (True, False), (True, True)])
def test_unmasked_rows_of_the_workspace_do_not_matter(B, R, keep, pair):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_2510_11683_gb300 as bg
    wl = Workload("padding_rows", B=B, P=2, R=R, H=136, V=700, n_t=4, G=1, t_mode=1, seed=5 + R,
                  targets="zipf", advantages="normal", eps_std=0.1)
    cpu = make_inputs(wl)
    o = oracle_run(wl, cpu)
    inp = {k: (v.cuda() if v is not None else None) for k, v in cpu.items()}
    ell_old = torch.from_numpy(o["ell_old"].T.astype(np.float32)).contiguous().cuda()
    prob = bg.problem_from(wl, keep_logits=keep, pair_dw=pair)

    def run(byte):
        ws = bg.alloc_workspace(prob)
        ws.fill_(byte)
        bg.clear_device_error(ws)
        ell = torch.empty((wl.n_t, B), device="cuda")
        coef, g = torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
        dX = torch.zeros((B, R, wl.H), device="cuda")
        dW = torch.zeros((wl.V, wl.H), device="cuda")
        for j in range(wl.n_t):
            bg.sample_mask(prob, j, ws)
            bg.elbo_fwd(prob, j, inp["X"], inp["W"], inp["Y"], ws, ell[j])
            bg.bound_coeffs(prob, j, ell[j], ell_old[j], inp["A"], coef, g, ws)
            bg.elbo_bwd_accumulate(prob, j, inp["X"], inp["W"], inp["Y"], coef, ws, dX, dW)
        assert bg.get_device_error(ws)[0] == 0
        return ell, dX, dW

    zero, ones = run(0), run(0xFF)
    for a, b in zip(zero, ones):
        assert torch.equal(a, b)
    ell, dX, dW = ones
    assert rel_ell_err(to64(ell).T, o["ell"]).max() <= 1e-3
    assert normwise(to64(dX), o["dX"]) <= 2e-2
    assert normwise(to64(dW), o["dW"]) <= 2e-2
