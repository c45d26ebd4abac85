"""The measured work of this framework: KL-NMF by the Diagonalized Newton Algorithm.

Every case is one call that a user's program repeats: a DNA iteration of one problem (dense
V, in each arithmetic form, or sparse V), a grouped iteration of many problems, or a
differentiable loss with its backward pass.  Sizes are those of the paper's Table 1 (ORL
and CMU PIE faces), of this repository's workloads (``workloads.py``) and of its tests.

The factors handed to a case are those of a factorisation under way: the usual starting
guess U(0.1, 1) (Section 4) after one DNA iteration in plain torch.  (Right at the starting
guess the two candidates of a column cost the same to rounding, so what the selection then
keeps says nothing about the code.)
"""
import functools
import math

import torch

import paper_1301_3389_gb300 as dna
from paper_1301_3389_gb300 import autograd

EPS, ALPHA = 0.01, 4.0   # the defaults of the options (Section 4)


# ------------------------------------------------------------------------------- cases
def _iterate(name, N, T, R, form, data="counts", **kw):
    return dict(name=name, kind="iterate", N=N, T=T, R=R, form=form, data=data, algo="dna",
                rho=0.0, lam=0.0, graph=True, **kw)


def listed():
    return [
        # a small matrix (the repository's smallest workload): every launch counts
        _iterate("small_f32", 256, 512, 16, "f32"),
        # ORL faces of Table 1, 4096 pixels x 165 images, the library's default engine
        _iterate("faces_orl_f32", 4096, 165, 80, "f32", data="pixels"),
        # CMU PIE faces of Table 1, 1024 x 11554 (T is not a multiple of 4)
        _iterate("faces_pie_f32", 1024, 11554, 80, "f32", data="pixels"),
        # the benchmark's counts matrix in the FP32 tensor-core form
        _iterate("counts_f32_tensor", 4096, 16384, 128, "f32t"),
        # the same in the BF16 form
        _iterate("counts_bf16", 4096, 16384, 128, "bf16"),
        # a ragged middle size of the tests above rank 256, FP32 tensor-core form
        _iterate("middle_rank300_f32_tensor", 2100, 2600, 300, "f32t", data="spectrogram"),
        # the largest workload: a spectrogram at rank 512, BF16 form
        _iterate("spectrogram_rank512_bf16", 8192, 32768, 512, "bf16", data="spectrogram"),
        # many uneven problems at once, in both forms of the batching calls
        dict(name="batched_bf16", kind="batched", count=128, form="bf16", n_max=2048, t_max=8192),
        dict(name="batched_f32", kind="batched", count=48, form="f32", n_max=2048, t_max=8192),
        # d_KL as a loss: forward and the gradients of V, W and H
        dict(name="kl_loss_f32", kind="loss", N=1024, T=4096, R=64),
        # an unrolled solve for H: forward, and back to V, W and H0 with a recomputed state
        # (two steps: float32 gradients through many say little, see the tests)
        dict(name="unrolled_f32", kind="unrolled", N=1024, T=4096, R=64, K=2, every=2),
        # term counts of the TDT2 shape (Section 4.2), sparse V
        dict(name="sparse_tdt2_f32", kind="sparse", N=36771, T=10212, R=64, density=0.0035),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sizes(rng, n, t, r, most):
    """N, T, R spread over the logarithms of their ranges, N T R at most ``most``."""
    while True:
        N, T, R = _log_int(rng, *n), _log_int(rng, *t), _log_int(rng, *r)
        if N * T * R <= most:
            return N, T, R


def draw(rng):
    kind = rng.choice(["f32", "f32", "f32t", "f32t", "bf16", "bf16", "batched", "loss",
                       "unrolled", "sparse"])
    if kind == "batched":
        form = rng.choice(["f32", "bf16"])
        return dict(kind="batched", count=_log_int(rng, 4, 96 if form == "bf16" else 32),
                    form=form, n_max=_log_int(rng, 256, 2048), t_max=_log_int(rng, 512, 8192))
    if kind == "loss":
        N, T, R = _sizes(rng, (64, 4096), (128, 16384), (8, 128), 1 << 31)
        return dict(kind="loss", N=N, T=T, R=R)
    if kind == "unrolled":
        N, T, R = _sizes(rng, (64, 2048), (128, 8192), (8, 128), 1 << 29)
        return dict(kind="unrolled", N=N, T=T, R=R, K=2, every=rng.randint(1, 2))
    if kind == "sparse":
        N, T, R = _sizes(rng, (1000, 36771), (500, 10212), (8, 128), 36771 * 10212 * 64)
        return dict(kind="sparse", N=N, T=T, R=R, density=rng.uniform(0.002, 0.01))
    # tensor-core ranks: up to the 300 of the tests, or the spectrogram's range
    ranks = (16, 300) if rng.random() < 0.75 else (400, 512)
    if kind == "f32":
        N, T, R = _sizes(rng, (64, 4096), (128, 16384), (8, 128), 1 << 32)
    elif kind == "f32t":
        N, T, R = _sizes(rng, (256, 8192), (512, 16384), ranks, 1 << 34)
    else:
        N, T, R = _sizes(rng, (256, 8192), (512, 32768), ranks, 1 << 36)
    reg = rng.random() < 0.25
    return dict(kind="iterate", N=N, T=T, R=R, form=kind,
                data=rng.choice(["counts", "pixels", "spectrogram"]),
                algo="mu" if rng.random() < 0.2 else "dna",
                rho=rng.uniform(0.01, 1.0) if reg else 0.0,
                lam=rng.uniform(0.01, 1.0) if reg else 0.0, graph=rng.random() < 0.75)


# ------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _gamma_half(g, *shape):
    """Gamma(1/2, 1) draws: half the square of a normal."""
    x = torch.randn(*shape, generator=g, device="cuda")
    return x.mul_(x).mul_(0.5)


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda").mul_(0.9).add_(0.1)


def _dense_v(g, N, T, R, data):
    """N x T data: Poisson counts of mean 2, pixel counts of mean 60, or a spectrogram of
    sparse activations over a small noise floor (no zeros)."""
    W0, H0 = _gamma_half(g, N, R), _gamma_half(g, R, T)
    if data == "spectrogram":
        H0.mul_(torch.rand(R, T, generator=g, device="cuda") >= 0.7)
        V = W0 @ H0
        return V.add_(torch.randn(N, T, generator=g, device="cuda").mul_(0.01).abs_())
    mean = {"counts": 2.0, "pixels": 60.0}[data]
    V = W0.mul_(mean / (0.25 * R)) @ H0
    return torch.poisson(V, generator=g)


# ----------------------------------------------------- Algorithm 1 in plain torch (any type)
def _ratios(V, Z):
    q = torch.where(V > 0, V / Z, torch.zeros_like(V))
    return q, torch.where(V > 0, q / Z, torch.zeros_like(V))


def _column_cost(V, Z):
    return (Z - torch.where(V > 0, V * torch.log(Z), torch.zeros_like(Z))).sum(0)


def _h_step(V, W, H, lam, algo="dna"):
    """Steps 2-15 for H at fixed W: per column the cheaper of the two candidates."""
    c = W.sum(0) + lam
    q, qb = _ratios(V, W @ H)
    a1 = (W.T @ q) / c[:, None]
    mu = H * a1
    if algo == "mu":
        return mu
    a, b = a1 - 1, ((W * W).T @ qb) / c[:, None]
    del q, qb
    hb = H * b
    down = H * torch.clamp_min(hb / torch.where(a < 0, hb - a, torch.ones_like(a)), EPS)
    step = torch.where(b > 0, a / torch.where(b > 0, b, torch.ones_like(b)), torch.zeros_like(b))
    nw = torch.where(a < 0, down, H + torch.minimum(step, ALPHA * H))
    den = c @ nw
    nw = nw * torch.where(den > 0, V.sum(0) / den, torch.ones_like(den))
    d_mu = _column_cost(V, W @ mu) + lam * mu.sum(0)
    d_nw = _column_cost(V, W @ nw) + lam * nw.sum(0)
    return torch.where(d_nw < d_mu, nw, mu)


def _iteration(V, W, H, rho, lam, algo="dna"):
    """Steps 4-29: H, step 16, W (the mirror on the transposes), step 29."""
    H = _h_step(V, W, H, lam, algo)
    s = H.sum(1) + rho
    H, W = H / s[:, None], W * s
    W = _h_step(V.T, H.T, W.T, rho, algo).T
    s = W.sum(0) + lam
    return W / s, H * s[:, None]


def _under_way(V, g, R, rho=0.0, lam=0.0):
    """The factors after one iteration from the starting guess (float32)."""
    W, H = _uniform(g, V.shape[0], R), _uniform(g, R, V.shape[1])
    s = W.sum(0) + lam
    W, H = _iteration(V, W / s, H * s[:, None], rho, lam)
    return W.contiguous(), H.contiguous()


def _iterate_inputs(c, seed):
    g = _generator(seed)
    V = _dense_v(g, c["N"], c["T"], c["R"], c["data"])
    return (V, *_under_way(V, g, c["R"], c["rho"], c["lam"]))


def _batched_inputs(c, seed):
    """V of each problem, and W, H of all of them as views of one buffer each.  Sizes are
    the case's, so another seed changes the values alone."""
    g = _generator(seed)
    Vs, Ws, Hs = [], [], []
    for N, T, R in _batched_sizes(c):
        V = _dense_v(g, N, T, R, "counts")
        W, H = _under_way(V, g, R)
        Vs.append(V), Ws.append(W), Hs.append(H)
    W, H = (torch.cat([x.reshape(-1) for x in xs]) for xs in (Ws, Hs))
    views = []
    for flat, xs in ((W, Ws), (H, Hs)):
        parts = torch.split(flat, [x.numel() for x in xs])
        views.append([p.view_as(x) for p, x in zip(parts, xs)])
    return Vs, W, H, views[0], views[1]


def _batched_sizes(c):
    """N and T log-uniform, R in {8, 16, 32, 64} (the repository's batched workload)."""
    g = torch.Generator()
    g.manual_seed(1000003 * c["count"] + 1009 * c["n_max"] + c["t_max"])
    u = torch.rand(c["count"], 3, generator=g, dtype=torch.float64).tolist()
    return [(int(64 * (c["n_max"] / 64) ** a), int(128 * (c["t_max"] / 128) ** b),
             (8, 16, 32, 64)[int(4 * r)]) for a, b, r in u]


def _sparse_inputs(c, seed):
    """Term counts with one dominant topic per document (Zipf vocabularies), as CSR."""
    g = _generator(seed)
    N, T, R = c["N"], c["T"], c["R"]
    want = c["density"] * N * T
    lens = torch.exp(0.8 * torch.randn(T, generator=g, device="cuda"))
    lens = torch.clamp((lens * (1.3 * want / float(lens.sum()))).round().long(), min=1)
    doc = torch.repeat_interleave(torch.arange(T, device="cuda"), lens)
    p = torch.arange(1, N + 1, device="cuda", dtype=torch.float64) ** -1.1
    cdf = torch.cumsum(p / p.sum(), 0)
    n = doc.numel()
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    rank = torch.clamp(torch.searchsorted(cdf, u), max=N - 1)
    perms = torch.stack([torch.randperm(N, generator=g, device="cuda") for _ in range(R + 1)])
    topic = torch.randint(0, R, (T,), generator=g, device="cuda")[doc]
    own = torch.rand(n, generator=g, device="cuda") < 0.7
    term = perms[torch.where(own, topic, torch.full_like(topic, R)), rank]
    key, cnt = torch.unique(term * T + doc, return_counts=True)   # sorted: rows are terms
    row_ptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(key // T, minlength=N), 0)
    vals = cnt.float()
    V = torch.zeros(N * T, device="cuda")
    V[key] = vals
    V = V.view(N, T)
    W, H = _under_way(V, g, R)
    return row_ptr, (key % T).to(torch.int32), vals, W, H, V


def _loss_inputs(c, seed):
    g = _generator(seed)
    V = _dense_v(g, c["N"], c["T"], c["R"], "counts")
    W, H = _under_way(V, g, c["R"])
    grad = torch.randn(c["R"], c["T"], generator=g, device="cuda") if c["kind"] == "unrolled" else None
    return V, W, H, grad


# ---------------------------------------------------------------------------- the calls
@functools.cache
def _stream():
    """The program's own stream (graph replay needs one that is not the default)."""
    return torch.cuda.Stream()


class _State:
    """Tensors and the library's handle of one case, released together."""

    def __init__(self, **kw):
        self.release = None
        self.__dict__.update(kw)

    def __del__(self):
        if self.release is not None:
            torch.cuda.synchronize()
            self.release()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("iterate", "sparse"):
        if kind == "iterate":
            V, W, H = _iterate_inputs(case, seed)
            form = {"f32": (dna.DNA_F32, dna.DNA_ENGINE_AUTO),
                    "f32t": (dna.DNA_F32, dna.DNA_ENGINE_TENSOR),
                    "bf16": (dna.DNA_BF16, dna.DNA_ENGINE_AUTO)}[case["form"]]
            opts = dna.make_opts(rho=case["rho"], lam=case["lam"], dtype=form[0], engine=form[1])
            ctx = dna.dna_create(case["N"], case["T"], case["R"], opts)
        else:
            row_ptr, col, vals, W, H, _ = _sparse_inputs(case, seed)
            V = (row_ptr, col, vals)
            ctx = dna.dna_create_sparse(case["N"], case["T"], case["R"], vals.numel())
        state = _State(case=case, V=V, W=W, H=H, ctx=ctx,
                       release=lambda: dna.dna_destroy(ctx))
        torch.cuda.synchronize()   # the inputs were made on another stream
        dna.dna_set_stream(ctx, _stream())
        if kind == "iterate":
            dna.dna_bind(ctx, V, W, H)
            dna.dna_use_graph(ctx, case["graph"])
        else:
            dna.dna_bind_csr(ctx, *V, W, H)
        return state
    if kind == "batched":
        Vs, W, H, Ws, Hs = _batched_inputs(case, seed)
        dtype = {"f32": dna.DNA_F32, "bf16": dna.DNA_BF16}[case["form"]]
        N, T, R = zip(*_batched_sizes(case))
        group = dna.dna_group_create(N, T, R, dna.make_opts(dtype=dtype))
        state = _State(case=case, V=Vs, W=W, H=H, views=(Ws, Hs), group=group,
                       release=lambda: dna.dna_group_destroy(group))
        torch.cuda.synchronize()
        dna.dna_group_set_stream(group)
        dna.dna_group_bind(group, Vs, Ws, Hs)
        dna.dna_group_use_graph(group, True)
        return state
    V, W, H, grad = _loss_inputs(case, seed)
    return _State(case=case, grad=grad, V=V.requires_grad_(), W=W.requires_grad_(),
                  H=H.requires_grad_())


def run(state):
    kind = state.case["kind"]
    if kind == "iterate":
        (dna.mu_iterate if state.case["algo"] == "mu" else dna.dna_iterate)(state.ctx, 1)
        return {"W": state.W, "H": state.H}
    if kind == "sparse":
        dna.dna_iterate(state.ctx, 1)
        return {"W": state.W, "H": state.H}
    if kind == "batched":
        dna.dna_group_iterate(state.group, 1)
        return {"W": state.W, "H": state.H}
    V, W, H = state.V, state.W, state.H
    if kind == "loss":
        loss = autograd.KLDiv.apply(V, W, H)
        dV, dW, dH = torch.autograd.grad(loss, (V, W, H))
        return {"loss": loss, "dV": dV, "dW": dW, "dH": dH}
    HK = autograd.UnrolledDNAH.apply(V, W, H, state.case["K"], state.case["every"])
    dV, dW, dH = torch.autograd.grad(HK, (V, W, H), state.grad)
    return {"H": HK, "dV": dV, "dW": dW, "dH": dH}


# ------------------------------------------------------------------------ what it takes
def _iteration_work(N, T, R, v_bytes, entries, algo="dna"):
    """V once, W and H read and written; 16 R flop per entry of V for DNA (the paper's
    count for an iteration, Section 3), 8 R for MU."""
    return {"bytes": v_bytes + 2 * 4 * R * (N + T),
            "flops": (16 if algo == "dna" else 8) * R * entries}


def work(case):
    kind = case["kind"]
    if kind == "batched":
        parts = [_iteration_work(N, T, R, 4 * N * T, N * T) for N, T, R in _batched_sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, T, R = case["N"], case["T"], case["R"]
    if kind == "iterate":
        return _iteration_work(N, T, R, 4 * N * T, N * T, case["algo"])
    if kind == "sparse":
        nnz = case["density"] * N * T
        return _iteration_work(N, T, R, 8 * nnz + 8 * N, nnz)
    if kind == "loss":   # z, W^t Q, Q H^t; V, W, H in and their gradients out
        return {"bytes": 2 * 4 * (N * T + R * (N + T)), "flops": 6 * R * N * T}
    # a step forward: z, A, B, two candidates' z (10 R); back: P1, P2, and two sums (H, W)
    # over s or o of each of its three factors (4 + 2 + 6)
    K = case["K"]
    return {"bytes": 2 * 4 * (N * T + R * (N + T)) + 4 * R * T, "flops": 22 * K * R * N * T}


# --------------------------------------------------------------------------- in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind in ("iterate", "sparse"):
        if kind == "iterate":
            V, W, H = _iterate_inputs(case, seed)
            rho, lam, algo = case["rho"], case["lam"], case["algo"]
        else:
            *_, W, H, V = _sparse_inputs(case, seed)
            rho, lam, algo = 0.0, 0.0, "dna"
        W, H = _iteration(V.double(), W.double(), H.double(), rho, lam, algo)
        return {"W": W, "H": H}
    if kind == "batched":
        Vs, _, _, Ws, Hs = _batched_inputs(case, seed)
        out = [_iteration(V.double(), W.double(), H.double(), 0.0, 0.0)
               for V, W, H in zip(Vs, Ws, Hs)]
        return {"W": torch.cat([w.reshape(-1) for w, _ in out]),
                "H": torch.cat([h.reshape(-1) for _, h in out])}
    V, W, H, grad = _loss_inputs(case, seed)
    V, W, H = V.double(), W.double(), H.double()
    if kind == "loss":
        Z = W @ H
        q, _ = _ratios(V, Z)
        log = torch.where(V > 0, torch.log(torch.where(V > 0, V, Z) / Z), torch.zeros_like(V))
        return {"loss": (V * log - V + Z).sum(), "dV": log, "dW": (1 - q) @ H.T,
                "dH": W.T @ (1 - q)}
    V.requires_grad_(), W.requires_grad_(), H.requires_grad_()
    HK = H
    for _ in range(case["K"]):
        HK = _unrolled_step(V, W, HK)
    dV, dW, dH = torch.autograd.grad(HK, (V, W, H), grad.double())
    return {"H": HK.detach(), "dV": dV, "dW": dW, "dH": dH}


def _unrolled_step(V, W, H):
    """_h_step with derivatives at v = 0 too (there q and qbar are still v / z, v / z^2)."""
    c = W.sum(0)
    Z = W @ H
    a1 = (W.T @ (V / Z)) / c[:, None]
    a, b = a1 - 1, ((W * W).T @ (V / (Z * Z))) / c[:, None]
    mu = H * a1
    hb = H * b
    down = H * torch.clamp_min(hb / torch.where(a < 0, hb - a, torch.ones_like(a)), EPS)
    nw = torch.where(a < 0, down, H + torch.minimum(a / b, ALPHA * H))
    nw = nw * (V.sum(0) / (c @ nw))
    with torch.no_grad():
        newton = _column_cost(V, W @ nw) < _column_cost(V, W @ mu)
    return torch.where(newton, nw, mu)
