"""Masks drawn in one round (before the wait for the kernel before) and in several.

The masking kernel holds up to 1,024 blocks of four positions, B ceil(R / 4),
in one round. On both sides of that line t, the masks and the ranks of the
masked rows are the oracle's, exactly, whatever the workspace held before.
"""
import numpy as np
import pytest

from oracle import bgpo_oracle as O
from synth import Workload
from tests.harness import ensure_built

pytestmark = pytest.mark.gpu

# (B, R): 1 block; 1,024 and 1,025 blocks of one sequence, of many, of four-position sequences
SIZES = [(1, 1), (1, 4096), (1, 4097), (4, 1021), (5, 820), (41, 97), (1024, 1), (1024, 4),
         (1025, 3)]


@pytest.mark.parametrize("B,R", SIZES)
@pytest.mark.parametrize("t_mode", [0, 1])
@pytest.mark.parametrize("lens", [False, True])
def test_draws_on_both_sides_of_one_round(B, R, t_mode, lens):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_2510_11683_gb300 as bg
    wl = Workload("mask_rounds", B=B, P=0, R=R, H=64, V=64, n_t=3, G=1, t_mode=t_mode, seed=B + R)
    resp_len = np.random.default_rng(R).integers(0, R + 1, size=B) if lens else None
    ts, masks = O.sample_masks(wl.seed, B, R, wl.n_t, t_mode, 7, resp_len)
    dev_len = torch.as_tensor(resp_len, dtype=torch.int32, device="cuda") if lens else None
    prob = bg.problem_from(wl, b_offset=7, resp_len=dev_len)
    ws = bg.alloc_workspace(prob)
    ws.fill_(0xFF)
    bg.clear_device_error(ws)
    t = torch.empty((wl.n_t, B), device="cuda")
    m = torch.full((wl.n_t, B, R), 9, dtype=torch.uint8, device="cuda")
    for j in range(wl.n_t):
        bg.sample_mask(prob, j, ws, t[j], m[j])
    assert bg.get_device_error(ws)[0] == 0
    assert np.array_equal(m.cpu().numpy(), masks.astype(np.uint8))
    assert np.array_equal(t.cpu().numpy(), ts.astype(np.float32))
    # the rows that the forward gathers: l of each sequence over its own masked rows
    X = torch.randn((B, R, wl.H), device="cuda").to(torch.bfloat16)
    W = torch.randn((wl.V, wl.H), device="cuda").to(torch.bfloat16)
    Y = torch.randint(0, wl.V, (B, R), dtype=torch.int32, device="cuda")
    ell = torch.empty(B, device="cuda")
    bg.elbo_fwd(prob, wl.n_t - 1, X, W, Y, ws, ell)
    ref = O.elbo_term(X.cpu().double().numpy(), W.cpu().double().numpy(), Y.cpu().numpy(), 0,
                      masks[-1], ts[-1])
    err = np.abs(ell.cpu().numpy() - ref) / np.maximum(np.abs(ref), 1.0)
    assert err.max() <= 1e-3
