"""Dependent launches keep stream order: blocks of a kernel may start while the
kernel before it still runs, but nothing is read or written before that kernel
has completed.

Hidden states, weights, targets and coefficients are rewritten by other kernels
of the stream immediately before and after every call, with no synchronisation;
the results must be the bits of the same calls with a synchronisation around
each.
"""
import pytest

from synth import CONFIGS, make_inputs
from tests.harness import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "ragged", "ragged_strat"])
@pytest.mark.parametrize("side_stream", [False, True])
def test_calls_see_what_the_stream_wrote_before_them(name, side_stream):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_2510_11683_gb300 as bg
    wl = CONFIGS[name]
    versions = [make_inputs(wl.with_(seed=wl.seed + 100 * k), device="cuda") for k in range(3)]
    prob = bg.problem_from(wl)

    def run(sync):
        def wait():
            if sync:
                torch.cuda.synchronize()

        ws = bg.alloc_workspace(prob)
        X, W, Y = (torch.zeros_like(versions[0][k]) for k in ("X", "W", "Y"))
        coef = torch.zeros(wl.B, device="cuda")
        out = []
        for step in range(6):
            v = versions[step % 3]
            j = step % wl.n_t
            dX = torch.zeros((wl.B, wl.R, wl.H), device="cuda")
            dW = torch.zeros((wl.V, wl.H), device="cuda")
            ell = torch.empty(wl.B, device="cuda")
            wait()
            bg.sample_mask(prob, j, ws)
            wait()
            X.copy_(v["X"])
            W.copy_(v["W"])
            Y.copy_(v["Y"])
            wait()
            bg.elbo_fwd(prob, j, X, W, Y, ws, ell)
            wait()
            torch.mul(ell, 1e-3, out=coef)
            wait()
            bg.elbo_bwd_accumulate(prob, j, X, W, Y, coef, ws, dX, dW)
            wait()
            kept = (ell.clone(), dX.clone(), dW.clone())
            X.fill_(float("nan"))
            W.fill_(float("nan"))
            Y.zero_()
            coef.fill_(float("nan"))
            out.append(kept)
        torch.cuda.synchronize()
        return out

    with torch.cuda.stream(torch.cuda.Stream() if side_stream else torch.cuda.default_stream()):
        want, got = run(True), run(False)
    for a, b in zip(want, got):
        for x, y in zip(a, b):
            assert torch.isfinite(x).all()
            assert torch.equal(x, y)
