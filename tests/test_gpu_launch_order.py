"""Dependent launches keep stream order: blocks of a kernel may start while the
kernel before it still runs, but nothing is read or written before that kernel
has completed.

Hidden states, weights, targets and coefficients are rewritten by other kernels
of the stream immediately before and after every call, with no synchronisation;
the results must be the bits of the same calls with a synchronisation around
each.
"""
import pytest

from synth import CONFIGS, Workload, make_inputs
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


@pytest.fixture(scope="module")
def sized():
    """A batch below and one above the size from which the backward's small kernels let
    the next kernel in late (2^23 response hidden values), three versions of each."""
    made = {}
    for key, kw in (("early", dict(B=4, R=130, H=320, V=3001)),
                    ("late", dict(B=8, R=512, H=2056, V=3001))):
        wl = Workload("order_" + key, P=2, n_t=2, G=2, t_mode=1, seed=7, **kw)
        assert (wl.B * wl.R * wl.H >= 1 << 23) == (key == "late")
        made[key] = wl, [make_inputs(wl.with_(seed=wl.seed + 100 * k), device="cuda")
                         for k in range(3)]
    return made


@pytest.mark.parametrize("size", ["early", "late"])
@pytest.mark.parametrize("flags", [{}, {"keep_logits": True}, {"pair_dw": True},
                                   {"vocab_chunk": 1280},
                                   {"keep_logits": True, "pair_dw": True, "vocab_chunk": 1280},
                                   {"keep_logits": True, "vocab_chunk": 1280}],
                         ids=["default", "kept", "paired", "chunked", "kept_paired_chunked",
                              "kept_chunked"])
def test_every_kernel_order_keeps_stream_order(sized, size, flags):
    """The kernel chains of every flag, on both sides of the early and late rule: a
    training loop's calls back to back, inputs overwritten around each."""
    import torch
    import paper_2510_11683_gb300 as bg
    ensure_built()
    wl, versions = sized[size]
    prob = bg.problem_from(wl, **flags)
    A = torch.linspace(-1, 1, wl.B, device="cuda")

    def run(sync):
        def wait():
            if sync:
                torch.cuda.synchronize()

        ws = bg.alloc_workspace(prob)
        X, W, Y = (torch.zeros_like(versions[0][k]) for k in ("X", "W", "Y"))
        coef, g = (torch.zeros(wl.B, device="cuda") for _ in range(2))
        out, plans = [], []
        for step in range(6):
            v, j = versions[step // 2], step % 2
            dX = torch.zeros((wl.B, wl.R, wl.H), device="cuda")
            dW = torch.zeros((wl.V, wl.H), device="cuda")
            ell, t = (torch.empty(wl.B, device="cuda") for _ in range(2))
            mask = torch.empty((wl.B, wl.R), dtype=torch.uint8, device="cuda")
            bg.sample_mask(prob, j, ws, t, mask)
            wait()
            X.copy_(v["X"])
            W.copy_(v["W"])
            Y.copy_(v["Y"])
            wait()
            bg.elbo_fwd(prob, j, X, W, Y, ws, ell)
            wait()
            bg.bound_coeffs(prob, j, ell, ell, A, coef, g, ws)
            wait()
            bg.elbo_bwd_accumulate(prob, j, X, W, Y, coef, ws, dX, dW)
            wait()
            X.fill_(float("nan"))
            W.fill_(float("nan"))
            Y.zero_()
            coef.fill_(float("nan"))
            out.append((t, mask, ell, g, dX.clone(), dW.clone()))
            plans.append(ws[20:24].clone())
        assert bg.get_device_error(ws) == (0, 0)
        return out, [int(p.view(torch.int32)) for p in plans]

    (want, splits), (got, _) = run(True), run(False)
    assert max(splits) > 1       # the split reduction runs
    for a, b in zip(want, got):
        for x, y in zip(a, b):
            assert torch.isfinite(x).all()
            assert torch.equal(x, y)


def test_forwards_without_a_workspace_keep_stream_order():
    import ctypes
    import torch
    import paper_2510_11683_gb300 as bg
    ensure_built()
    # one mask round (draws before the wait) and several
    for R in (130, 2100):
        wl = Workload("order_noalloc", B=4, P=2, R=R, H=128, V=777, n_t=2, G=2, t_mode=0, seed=9)
        versions = [make_inputs(wl.with_(seed=wl.seed + 100 * k), device="cuda") for k in range(3)]
        prob = bg.problem_from(wl)

        def run(sync):
            X, W, Y = (torch.zeros_like(versions[0][k]) for k in ("X", "W", "Y"))
            out = []
            for step in range(6):
                v = versions[step % 3]
                t, ell = (torch.empty(wl.B, device="cuda") for _ in range(2))
                X.copy_(v["X"])
                W.copy_(v["W"])
                Y.copy_(v["Y"])
                if sync:
                    torch.cuda.synchronize()
                bg._lib.check("bgpo_elbo_fwd_noalloc", bg._lib.lib().bgpo_elbo_fwd_noalloc(
                    ctypes.byref(prob), step % 2, X.data_ptr(), W.data_ptr(), Y.data_ptr(),
                    t.data_ptr(), ell.data_ptr(), torch.cuda.current_stream().cuda_stream))
                if sync:
                    torch.cuda.synchronize()
                X.fill_(float("nan"))
                W.fill_(float("nan"))
                Y.zero_()
                out.append((t, ell))
            torch.cuda.synchronize()
            return out

        for a, b in zip(run(True), run(False)):
            for x, y in zip(a, b):
                assert torch.isfinite(x).all()
                assert torch.equal(x, y)
