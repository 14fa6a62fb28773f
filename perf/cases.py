"""Workloads of the BGPO LM-head ELBO path, for measuring it.

A case is one pass of a user's program through the calls of the package:

  step     Algorithm 1's inner loops over one batch: the group advantages (when
           the batch holds whole groups), then for every MC sample j masking,
           ELBO forward, bound coefficients and accumulated backward
  old      the old policy's forward-only pass over every MC sample (Eq. 10)
  vrpo     the objective the bound replaces (Eq. 7), its forwards run twice
  noalloc  one sample's forward on the library's own scratch

Sizes and options of a case:

  B, P, R  responses, prompt and response length;  H, V  the LM head
  n_t, G   MC samples per response, group size;  strat  stratified t
  keep     BGPO_FLAG_KEEP_LOGITS;  pair  BGPO_FLAG_PAIR_DW
  chunk    columns of the vocabulary the backward handles at a time (0: default)
  own_x    each MC sample has its own hidden states (and its own dX), as when the
           network sees each masked sequence
  ragged   responses of different lengths (resp_len)
"""
import ctypes
import math

import numpy as np
import torch

import paper_2510_11683_gb300 as bg

EPS_STD = 0.1      # spread of l_old around l (log-ratio of the two policies)
ZIPF_S = 1.1


def _case(kind, B, P, R, H, V, n_t, G, strat=False, keep=False, pair=False, chunk=0, own_x=False,
          ragged=False, name=None):
    c = dict(kind=kind, B=B, P=P, R=R, H=H, V=V, n_t=n_t, G=G, strat=strat, keep=keep, pair=pair,
             chunk=chunk, own_x=own_x, ragged=ragged)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a toy head, as in a unit test or a method study: every launch is short
        _case("step", 2, 16, 32, 64, 512, 4, 2, name="step_toy"),
        # a small head with ragged sizes in every dimension, padded responses, logits kept
        _case("step", 5, 3, 130, 320, 777, 5, 5, strat=True, keep=True, ragged=True,
              name="step_small_ragged"),
        # a log-likelihood asked for by a process that cannot allocate device memory
        _case("noalloc", 4, 32, 128, 1024, 8192, 4, 4, name="ell_noalloc"),
        # a small model's head; the network runs on each masked sequence
        _case("step", 8, 64, 128, 2048, 32000, 4, 8, own_x=True, ragged=True, name="step_32k"),
        # the comparison objective on a mid-sized head with an odd vocabulary
        _case("vrpo", 6, 37, 333, 1536, 50001, 2, 6, name="vrpo_50k_odd"),
        # a batch of one response per micro-step, as where the network fills the memory
        _case("step", 1, 128, 256, 4096, 126464, 2, 8, strat=True, pair=True, own_x=True,
              name="step_8b_one_response"),
        # the same head with very few response tokens: W and dW traffic alone
        _case("step", 2, 8, 24, 4096, 126464, 1, 2, name="step_8b_few_rows"),
        # the old policy's l for one group of 8 responses of 256 tokens
        _case("old", 8, 128, 256, 4096, 126464, 2, 8, name="old_8b_r256"),
        # two MC samples of a training step on the same batch, dW paired
        _case("step", 8, 128, 256, 4096, 126464, 2, 8, strat=True, pair=True,
              name="step_8b_r256_paired"),
        # responses of 512, logits kept
        _case("step", 8, 256, 512, 4096, 126464, 2, 8, strat=True, keep=True, pair=True,
              name="step_8b_r512_kept"),
        # 16 responses of 512 with the library's default flags: the backward in chunks
        _case("step", 16, 256, 512, 4096, 126464, 2, 8, strat=True, name="step_8b_r512_chunked"),
        # the largest batch: 32 responses of 1024 on a 7B-sized head
        _case("step", 32, 512, 1024, 3584, 152064, 1, 8, name="step_7b_r1024"),
    ]


_LARGEST = 32 * 1024 * 3584 * 152064   # B R H V n_t of the largest listed case


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _noalloc_bytes(c):
    m_pad = -(-c["B"] * c["R"] // 256) * 256
    return m_pad * (2 * c["H"] + 8 * -(-c["V"] // 256) + 20) + 16 * c["B"] + 12288


def draw(rng):
    while True:
        kind = rng.choice(["step", "step", "step", "step", "old", "old", "vrpo", "noalloc"])
        B, R = _log_int(rng, 1, 32), _log_int(rng, 16, 1024)
        H, V = 8 * _log_int(rng, 8, 512), _log_int(rng, 512, 152064)
        if V > 4096 and rng.random() < 0.5:
            V = V // 64 * 64                     # heads are often padded to a multiple of 64
        G = rng.choice([g for g in (1, 2, 3, 4, 5, 6, 8) if B % g == 0 and g > 1] or [8])
        step = kind == "step"
        c = _case(kind, B, rng.choice([0, 5, 32, 128, 512]), R, H, V, rng.choice([1, 2, 3, 4]), G,
                  strat=rng.random() < 0.4, keep=step and rng.random() < 0.3,
                  pair=step and rng.random() < 0.4,
                  chunk=256 * rng.randint(8, 64) if step and rng.random() < 0.15 else 0,
                  own_x=step and rng.random() < 0.3, ragged=rng.random() < 0.3)
        if kind == "noalloc" and _noalloc_bytes(c) > 30 << 20:
            continue
        if B * R * H * V * c["n_t"] <= _LARGEST and B * R <= 16384:
            return c


# ---- inputs -----------------------------------------------------------------------


def _inputs(case, seed):
    """What the seed alone decides, on the GPU (and the Philox key and lengths as numbers)."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)
    B, P, R, H, V, n_t = (case[k] for k in ("B", "P", "R", "H", "V", "n_t"))

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    d = {"key": (int(seed) * 0x9E3779B97F4A7C15 + 1) % (1 << 64)}
    d["X"] = normal(*((n_t,) if case["own_x"] else ()), B, P + R, H).to(torch.bfloat16)
    W = torch.empty((V, H), dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 28) // H)
    for v in range(0, V, rows):
        n = min(rows, V - v)
        W[v:v + n] = normal(n, H) * H ** -0.5
    d["W"] = W
    cdf = torch.arange(1, V + 1, dtype=torch.float64, device="cuda").pow(-ZIPF_S).cumsum(0)
    u = torch.rand((B, R), generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    d["Y"] = torch.searchsorted(cdf, u).clamp_(max=V - 1).to(torch.int32)
    d["eps"] = EPS_STD * normal(n_t, B)
    d["reward"] = normal(B)                     # advantages themselves where B is no whole group
    d["lens"] = None
    if case["ragged"]:
        lo = max(1, R // 4)
        d["lens"] = torch.randint(lo, R + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    return d


def _grouped(case):
    return case["G"] > 1 and case["B"] % case["G"] == 0


def _problem(case, d, keep, pair):
    return bg.problem(case["B"], case["P"], case["R"], case["H"], case["V"], case["n_t"], case["G"],
                      t_mode=bg.T_STRATIFIED if case["strat"] else bg.T_IID, seed=d["key"],
                      resp_len=d["lens"], keep_logits=keep, pair_dw=pair,
                      vocab_chunk=case["chunk"])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind, B, R, H, V, n_t = (case[k] for k in ("kind", "B", "R", "H", "V", "n_t"))
    f32 = dict(dtype=torch.float32, device="cuda")
    s["prob"] = _problem(case, s, case["keep"], case["pair"])
    s["ell"] = torch.empty((n_t, B), **f32)
    if kind == "noalloc":
        s["t"], s["ell"] = torch.empty(B, **f32), torch.empty(B, **f32)
        return s
    s["ws"] = bg.alloc_workspace(s["prob"])
    if kind == "old":
        s["t"] = torch.empty((n_t, B), **f32)
        s["mask"] = torch.empty((n_t, B, R), dtype=torch.uint8, device="cuda")
        return s
    # the old policy's l, from its own pass before the step: here l of this policy + eps
    fwd = _problem(case, s, False, False)
    ws = bg.alloc_workspace(fwd)
    s["ell_old"] = torch.empty((n_t, B), **f32)
    for j in range(n_t):
        bg.sample_mask(fwd, j, ws)
        bg.elbo_fwd(fwd, j, _x(s, j), s["W"], s["Y"], ws, s["ell_old"][j])
    s["ell_old"] += s["eps"]
    s["A"] = torch.empty(B, **f32) if _grouped(case) else s["reward"]
    s["coef"] = torch.empty((n_t, B) if kind == "step" else (B,), **f32)
    s["g"] = torch.empty((n_t, B) if kind == "step" else (B,), **f32)
    s["dX"] = torch.empty(((n_t,) if case["own_x"] else ()) + (B, R, H), **f32)
    s["dW"] = torch.empty((V, H), **f32)
    return s


def _x(s, j):
    return s["X"][j] if s["case"]["own_x"] else s["X"]


def run(s):
    case = s["case"]
    prob, n_t = s["prob"], case["n_t"]
    W, Y, ell = s["W"], s["Y"], s["ell"]
    if case["kind"] == "noalloc":
        st = bg._lib.lib().bgpo_elbo_fwd_noalloc(
            ctypes.byref(prob), 0, s["X"].data_ptr(), W.data_ptr(), Y.data_ptr(),
            s["t"].data_ptr(), ell.data_ptr(), torch.cuda.current_stream().cuda_stream)
        bg._lib.check("bgpo_elbo_fwd_noalloc", st)
        return {"t": s["t"], "ell": ell}
    ws = s["ws"]
    if case["kind"] == "old":
        for j in range(n_t):
            bg.sample_mask(prob, j, ws, s["t"][j], s["mask"][j])
            bg.elbo_fwd(prob, j, s["X"], W, Y, ws, ell[j])
        return {"t": s["t"], "mask": s["mask"], "ell": ell}
    A, coef, g, dX, dW = s["A"], s["coef"], s["g"], s["dX"], s["dW"]
    dX.zero_()
    dW.zero_()
    if _grouped(case):
        bg.group_advantage(prob, s["reward"], A)
    if case["kind"] == "vrpo":
        for j in range(n_t):
            bg.sample_mask(prob, j, ws)
            bg.elbo_fwd(prob, j, s["X"], W, Y, ws, ell[j])
        bg.vrpo_coeffs(prob, ell, s["ell_old"], A, coef, g, ws)
        for j in range(n_t):
            bg.sample_mask(prob, j, ws)
            bg.elbo_fwd(prob, j, s["X"], W, Y, ws, ell[j])
            bg.elbo_bwd_accumulate(prob, j, s["X"], W, Y, coef, ws, dX, dW)
    else:
        for j in range(n_t):
            X = _x(s, j)
            bg.sample_mask(prob, j, ws)
            bg.elbo_fwd(prob, j, X, W, Y, ws, ell[j])
            bg.bound_coeffs(prob, j, ell[j], s["ell_old"][j], A, coef[j], g[j], ws)
            bg.elbo_bwd_accumulate(prob, j, X, W, Y, coef[j], ws, dX[j] if case["own_x"] else dX,
                                   dW)
    return {"ell": ell, "coef": coef, "g": g, "dX": dX, "dW": dW}


# ---- what a pass cannot do without ---------------------------------------------------


def work(case):
    """t is uniform on (0, 1]: half of the response positions are masked in the mean."""
    B, R, H, V, n_t = (case[k] for k in ("B", "R", "H", "V", "n_t"))
    samples = 1 if case["kind"] == "noalloc" else n_t
    len_ = 0.625 * R if case["ragged"] else R
    rows = 0.5 * B * len_ * samples
    read = 2 * V * H + 2 * H * (rows if case["own_x"] or samples == 1 else B * len_) + 4 * B * R
    if case["kind"] in ("old", "noalloc"):
        return {"bytes": read + 8 * samples * B, "flops": 2 * rows * H * V}
    written = 4 * V * H + 4 * B * R * H * (n_t if case["own_x"] else 1)
    return {"bytes": read + written, "flops": 6 * rows * H * V}


def tolerance(case):
    # l: fp32 sums of bf16 products; measured 1e-7 to 2.2e-6 from the 64-bit values.
    # Gradients: dL/dz is rounded to bf16 (2^-9 an element) before two contractions; measured
    # 0.7e-3 to 1.9e-3 from the 64-bit values. Each limit is four times the largest.
    return {"rel": 8e-6} if case["kind"] in ("old", "noalloc") else {"rel": 7.5e-3}


# ---- the same values in 64 bits ------------------------------------------------------

_MASK32 = np.uint64(0xFFFFFFFF)


def _mulhilo(a, b):
    """High and low words of the 128-bit products of a constant and an array."""
    a0, a1 = np.uint64(a & 0xFFFFFFFF), np.uint64(a >> 32)
    b0, b1 = b & _MASK32, b >> np.uint64(32)
    lo = a0 * b0
    m1 = a1 * b0 + (lo >> np.uint64(32))
    m2 = a0 * b1 + (m1 & _MASK32)
    hi = a1 * b1 + (m1 >> np.uint64(32)) + (m2 >> np.uint64(32))
    return hi, (m2 << np.uint64(32)) | (lo & _MASK32)


def _philox(c0, c1, c2, c3, key):
    """Philox4x64-10 (Salmon et al., SC 2011) on arrays of counters; key (key, 0)."""
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = key, 0
    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0 = _mulhilo(0xD2E7470EE14C6C93, c[0])
            h1, l1 = _mulhilo(0xCA5A826395121157, c[2])
            c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
            k0 = (k0 + 0x9E3779B97F4A7C15) % (1 << 64)
            k1 = (k1 + 0xBB67AE8584CAA73B) % (1 << 64)
    return c


def _draws(case, key, lens, j):
    """t [B] in 64 bits and the mask [B, R] of MC sample j."""
    B, R, n_t = case["B"], case["R"], case["n_t"]
    b = np.arange(B, dtype=np.uint64)
    u = _philox(0, b, j, 1, key)[0] >> np.uint64(40)
    D = n_t if case["strat"] else 1                       # in units of 2^24
    T = u + np.uint64(1 + ((j << 24) if case["strat"] else 0))
    q = np.arange(-(-R // 4), dtype=np.uint64)
    words = np.stack(_philox(q[None, :], b[:, None], j, 0, key), axis=-1).reshape(B, -1)[:, :R]
    mask = (words >> np.uint64(40)) * np.uint64(D) < T[:, None]
    if lens is not None:
        mask &= np.arange(R)[None, :] < lens.cpu().numpy()[:, None]
    return T.astype(np.float64) / float(D << 24), mask


def exact(case, seed):
    B, P, R, H, V, n_t, kind = (case[k] for k in ("B", "P", "R", "H", "V", "n_t", "kind"))
    passes = {"step": 3, "vrpo": 4}.get(kind, 1)
    if passes * B * R * n_t * H * V > 8e12:               # over about 20 s in 64 bits
        return None
    d = _inputs(case, seed)
    W = d["W"].double()

    def forward(j):
        t, mask = _draws(case, d["key"], d["lens"], j)
        t = torch.from_numpy(t).cuda()
        bi = torch.from_numpy(np.argwhere(mask)).cuda()
        x = (d["X"][j] if case["own_x"] else d["X"])[bi[:, 0], P + bi[:, 1]].double()
        y = d["Y"][bi[:, 0], bi[:, 1]].long()
        z = x @ W.T
        lse = torch.logsumexp(z, 1)
        logp = z.gather(1, y[:, None])[:, 0] - lse
        ell = torch.zeros(B, dtype=torch.float64, device="cuda").index_add_(0, bi[:, 0], logp) / t
        return t, mask, bi, x, y, z, lse, ell

    if kind in ("old", "noalloc"):
        got = [forward(j) for j in range(1 if kind == "noalloc" else n_t)]
        t, ell = torch.stack([f[0] for f in got]), torch.stack([f[7] for f in got])
        if kind == "noalloc":
            return {"t": t[0], "ell": ell[0]}
        return {"t": t, "mask": torch.from_numpy(np.stack([f[1] for f in got])).to(torch.uint8),
                "ell": ell}

    A = d["reward"].double()
    if _grouped(case):
        r = A.view(-1, case["G"])
        A = ((r - r.mean(1, keepdim=True)) / r.std(1, keepdim=True, unbiased=False)).reshape(-1)
    scale = -1.0 / case["G"] / n_t
    eps = d["eps"].double()
    dX = torch.zeros(((n_t,) if case["own_x"] else ()) + (B, R, H), dtype=torch.float64,
                     device="cuda")
    dW = torch.zeros((V, H), dtype=torch.float64, device="cuda")
    ells, coefs, gs = [], [], []
    if kind == "vrpo":                                    # d = -eps in every sample
        e = torch.exp(-eps.mean(0))
        coef, g = scale * A * e, e * A
    for j in range(n_t):
        t, _, bi, x, y, z, lse, ell = forward(j)
        if kind == "step":
            e = torch.where(A >= 0, 1.0, torch.exp(-eps[j]))
            coef = scale * A * e
            gs.append(torch.where(A >= 0, 1 - eps[j], e) * A / n_t)
            coefs.append(coef)
        ells.append(ell)
        w = (coef / t)[bi[:, 0]]
        z.sub_(lse[:, None]).exp_().mul_(-w[:, None])
        z[torch.arange(len(y), device="cuda"), y] += w
        (dX[j] if case["own_x"] else dX)[bi[:, 0], bi[:, 1]] += z @ W
        dW.addmm_(z.T, x)
        del z
    if kind == "step":
        coef, g = torch.stack(coefs), torch.stack(gs)
    return {"ell": torch.stack(ells), "coef": coef, "g": g, "dX": dX, "dW": dW}
