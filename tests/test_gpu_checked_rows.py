"""The checked build's bound on the row count, in the backward.

After a good backward the row count in the workspace's error word is set past
the batch's positions and the backward runs again: every kernel must skip its
work (the split reduction too, whose flat forms walk as many tiles as the count
asks for), the transpose reports BGPO_ERR_BOUNDS first, and dX and dW keep their
bits. Hidden sizes on both sides of the reduction's row form, split plans.
"""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from tests.harness import ensure_built  # noqa: E402

ERR_M, ERR_DX_SPLITS = 3, 5      # words of the error word (csrc/bgpo_plan.h)
KID_XM_TRANSPOSE = 14


def _child():
    import torch
    import paper_2510_11683_gb300 as bg
    from paper_2510_11683_gb300 import _lib
    from synth import Workload, make_inputs

    assert _lib.lib_path().endswith("libbgpo_checked.so")
    out = []
    for H in (200, 1024, 2056):
        wl = Workload("checked_rows", B=2, P=1, R=150, H=H, V=3000, n_t=2, G=1, t_mode=1, seed=5,
                      targets="zipf", advantages="normal", eps_std=0.1)
        inp = make_inputs(wl, device="cuda")
        prob = bg.problem_from(wl)
        ws = bg.alloc_workspace(prob)
        word = ws[:64].view(torch.int32)
        ell = torch.empty(wl.B, device="cuda")
        coef = torch.full((wl.B,), 0.1, device="cuda")
        dX = torch.zeros((wl.B, wl.R, wl.H), device="cuda")
        dW = torch.zeros((wl.V, wl.H), device="cuda")
        args = (inp["X"], inp["W"], inp["Y"], coef, ws, dX, dW)
        bg.sample_mask(prob, 1, ws)
        bg.elbo_fwd(prob, 1, inp["X"], inp["W"], inp["Y"], ws, ell)
        bg.elbo_bwd_accumulate(prob, 1, *args)
        good = bg.get_device_error(ws)
        splits = int(word[ERR_DX_SPLITS])
        kept = dX.clone(), dW.clone()
        word[ERR_M] = wl.B * wl.R + 1
        bg.elbo_bwd_accumulate(prob, 1, *args)
        out.append({"H": H, "good": good, "splits": splits, "error": bg.get_device_error(ws),
                    "grads": bool(kept[0].any() and kept[1].any()),
                    "kept": bool(torch.equal(dX, kept[0]) and torch.equal(dW, kept[1]))})
    print(json.dumps(out))


@pytest.mark.gpu
def test_a_row_count_past_the_batch_is_reported_and_adds_nothing():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built(checked=True)
    env = dict(os.environ, BGPO_LIBRARY="checked", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    for c in json.loads(r.stdout.strip().splitlines()[-1]):
        assert c["good"] == [0, 0] and c["splits"] > 1 and c["grads"], c
        assert c["error"] == [9, KID_XM_TRANSPOSE * 16 + 9] and c["kept"], c


if __name__ == "__main__":
    _child()
