"""The work users of this framework have it do, as cases that can be timed and compared.

Each case goes through the public entry points of paper_2311_07710_gb300.pdqp: whole solves
(single problems in both precisions, batches, a parameterised family, a low-rank objective),
the relative KKT error of a control loop, and the learned warm start (fit, training, inference,
and the tensor-core GEMM it runs on).  Problems are seeded synthetic instances of the shapes
this repository documents, assembled on the GPU.
"""
import math

import numpy as np
import torch

from paper_2311_07710_gb300 import pdqp

NX, NU = 12, 4                      # states and inputs of the control problems
DEV = "cuda"
F64, I32 = torch.float64, torch.int32


def listed():
    return [
        # one relKKT evaluation inside a real-time control loop: the smallest call, all latency
        dict(name="kkt_control_loop", kind="kkt", horizon=10),
        # a small sparse problem solved on its own, to tolerance: launches and barriers count
        dict(name="qp_n1000_mixed", kind="qp", n=1000, m=500, q_per_row=5, a_per_row=10, precision="mixed"),
        # the default workload: a large sparse problem on a kept handle
        dict(name="qp_n1e6_mixed", kind="large", n=1_000_000, m=500_000, precision="mixed"),
        # plain float64, the precision by default, at an odd middle size
        dict(name="qp_n300007_fp64", kind="large", n=300_007, m=150_003, precision="fp64"),
        # a batch of control problems of uneven horizons, each batch new: create, solve, destroy
        dict(name="control_batch_4096_mixed", kind="batch", count=4096, t_lo=10, t_hi=100, precision="mixed"),
        # a few control problems in plain float64
        dict(name="control_batch_77_fp64", kind="batch", count=77, t_lo=10, t_hi=100, precision="fp64"),
        # members of a parameterised family on one handle, from the all-zero start
        dict(name="family_300_mixed", kind="family", n=20_000, m=10_000, count=300, precision="mixed"),
        # a portfolio with a dense low-rank factor and two dense rows
        dict(name="portfolio_n1e5_r64_mixed", kind="portfolio", n=100_000, r=64, precision="mixed"),
        # normalisation fitted to a training set of solver outputs
        dict(name="ws_fit_4096", kind="fit", n=20_000, m=10_000, count=4096),
        # one epoch of training on such a set
        dict(name="ws_train_2048", kind="train", n=20_000, m=10_000, width=1024, depth=3, count=2048, batch=256),
        # warm starts predicted for one family handle
        dict(name="ws_infer_2048", kind="infer", n=20_000, m=10_000, width=1024, depth=3, count=2048),
        # the raw tensor-core GEMM at its benchmark size
        dict(name="gemm_8192", kind="gemm", M=8192, N=8192, K=8192, epilogue="plain"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kkt", "qp", "large", "batch", "family", "portfolio", "fit", "train", "infer", "gemm"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if kind == "kkt":
        return dict(kind=kind, horizon=_log(rng, 10, 3000))
    if kind == "qp":
        n = _log(rng, 200, 10_000)
        return dict(kind=kind, n=n, m=max(1, n // rng.choice([1, 2, 3])), q_per_row=rng.randint(2, 5),
                    a_per_row=rng.randint(4, 12), precision=precision)
    if kind == "large":
        n = _log(rng, 20_000, 1_000_000)
        return dict(kind=kind, n=n, m=n // 2, precision="mixed" if n > 600_000 else precision)
    if kind == "batch":
        lo = rng.randint(5, 40)
        return dict(kind=kind, count=_log(rng, 2, 4000), t_lo=lo, t_hi=lo + rng.randint(0, 60), precision="mixed")
    if kind == "family":
        n = _log(rng, 400, 20_000)
        return dict(kind=kind, n=n, m=n // 2, count=_log(rng, 3, 300), precision=precision if n < 4000 else "mixed")
    if kind == "portfolio":
        return dict(kind=kind, n=_log(rng, 2000, 100_000), r=rng.choice([8, 16, 24, 33, 64]), precision="mixed")
    n = _log(rng, 400, 20_000)
    if kind == "fit":
        return dict(kind=kind, n=n, m=n // 2 + 1, count=_log(rng, 50, 4096))
    if kind in ("train", "infer"):
        batch = 8 * rng.randint(4, 32)
        case = dict(kind=kind, n=n, m=n // 2 + 1, width=rng.choice([256, 512, 1024]), depth=rng.randint(1, 3),
                    count=_log(rng, 256, 2048))
        return dict(case, batch=batch) if kind == "train" else case
    return dict(kind=kind, M=_log(rng, 64, 8192), N=_log(rng, 64, 8192), K=8 * _log(rng, 8, 1024),
                epilogue=rng.choice(["plain", "bias_relu_bf16"]))


# --------------------------------------------------------------------------
# problems
# --------------------------------------------------------------------------
def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1_000_003 + salt) % (2 ** 62))


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def _csr(row, col, val, rows, cols):
    """CSR (int32 row pointers and columns) of distinct coordinates."""
    order = torch.argsort(row * cols + col)
    rp = torch.zeros(rows + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=rows), 0)
    return rp.to(I32), col[order].to(I32), val[order].contiguous()


def _row_sums(csr, v):
    rp, col, val = csr
    prod = val * v[col.long()] if v is not None else val.abs()
    return torch.segment_reduce(prod, "sum", lengths=(rp[1:] - rp[:-1]).long(), initial=0.0)


def _entries_per_row(g, rows, cols, k):
    """Up to k distinct uniform columns in each of `rows` rows (drawn duplicates fall away)."""
    c = torch.sort(torch.randint(0, cols, (rows, min(k, cols)), generator=g, device=DEV), 1).values
    keep = torch.ones_like(c, dtype=torch.bool)
    keep[:, 1:] = c[:, 1:] != c[:, :-1]
    r = torch.arange(rows, device=DEV)[:, None].expand_as(c)
    return r[keep], c[keep]


def _rhs(g, A, m, m_eq, n):
    """b with a feasible point: exact on the equality rows, slack U(0, 1) on the others."""
    b = _row_sums(A, _uniform(g, -1.0, 1.0, n))
    b[m_eq:] -= _uniform(g, 0.0, 1.0, m - m_eq)
    return b


def _box(n, lo, hi):
    return torch.full((n,), lo, device=DEV, dtype=F64), torch.full((n,), hi, device=DEV, dtype=F64)


def _gram_qp(seed, n, m, q_per_row, a_per_row):
    """Q = B'B + 0.01 I and A with a few N(0, 1) entries per row; c ~ N(0, 1); box [-10, 10]."""
    g = _gen(seed, 1)
    ar, ac = _entries_per_row(g, m, n, a_per_row)
    A = _csr(ar, ac, _normal(g, ar.numel()), m, n)
    # Q from the pairs of entries of each row of B, summed in a fixed order on the host
    br, bc = _entries_per_row(g, n, n, q_per_row)
    bv = _normal(g, br.numel()).cpu().numpy()
    br, bc = br.cpu().numpy(), bc.cpu().numpy()
    start = np.searchsorted(br, np.arange(n + 1))
    per = np.diff(start)
    left = np.repeat(np.arange(br.size), per[br])
    first = np.cumsum(per[br]) - per[br]
    right = start[br[left]] + np.arange(left.size) - np.repeat(first, per[br])
    key = np.concatenate([bc[left] * n + bc[right], np.arange(n) * (n + 1)])
    val = np.concatenate([bv[left] * bv[right], np.full(n, 0.01)])
    order = np.argsort(key, kind="stable")
    key, val = key[order], val[order]
    head = np.flatnonzero(np.concatenate([[True], key[1:] != key[:-1]]))
    key, val = torch.from_numpy(key[head]).to(DEV), torch.from_numpy(np.add.reduceat(val, head)).to(DEV)
    Q = _csr(key // n, key % n, val, n, n)
    l, u = _box(n, -10.0, 10.0)
    return dict(n=n, m=m, m_eq=m // 2, Q=Q, A=A, c=_normal(g, n), b=_rhs(g, A, m, m // 2, n), l=l, u=u)


def _large_qp(seed, n, m):
    """Ten entries per column of A at uniform rows; Q a dominated diagonal with about five
    mirrored off-diagonal entries per row; box [-10, 10]."""
    g = _gen(seed, 2)
    ac, ar = _entries_per_row(g, n, m, 10)
    A = _csr(ar, ac, _normal(g, ar.numel()), m, n)
    i = torch.randint(0, n, (n * 5 // 2,), generator=g, device=DEV)
    j = torch.randint(0, n, (n * 5 // 2,), generator=g, device=DEV)
    key = torch.unique((torch.minimum(i, j) * n + torch.maximum(i, j))[i != j])
    i, j = key // n, key % n
    v = 0.1 * _normal(g, i.numel())
    d = torch.arange(n, device=DEV)
    dominant = _row_sums(_csr(torch.cat([i, j]), torch.cat([j, i]), torch.cat([v, v]), n, n), None)
    Q = _csr(torch.cat([i, j, d]), torch.cat([j, i, d]), torch.cat([v, v, _uniform(g, 0.1, 10.0, n) + dominant]), n, n)
    l, u = _box(n, -10.0, 10.0)
    return dict(n=n, m=m, m_eq=m // 2, Q=Q, A=A, c=_normal(g, n), b=_rhs(g, A, m, m // 2, n), l=l, u=u)


def _control_qps(seed, count, t_lo, t_hi):
    """`count` control problems stacked block-diagonally: variables (x_0..x_T, u_0..u_{T-1}),
    rows x_0 = x_init and x_{t+1} - A_d x_t - B_d u_t = 0, |x| <= 5, |u| <= 1, Q diagonal;
    redrawn until the uncontrolled trajectory stays inside its bounds."""
    T = np.random.default_rng((count, t_lo, t_hi)).integers(t_lo, t_hi + 1, count)   # the sizes are the case's
    rng = np.random.default_rng((int(seed), 3))
    Ad, Bd, x0 = np.empty((count, NX, NX)), np.empty((count, NX, NU)), np.empty((count, NX))
    todo = np.arange(count)
    while todo.size:
        a = np.eye(NX) + 0.1 * rng.standard_normal((todo.size, NX, NX))
        a /= np.maximum(1.0, np.abs(np.linalg.eigvals(a)).max(1))[:, None, None]
        x = rng.uniform(-1.0, 1.0, (todo.size, NX))
        Ad[todo], Bd[todo], x0[todo] = a, 0.1 * rng.standard_normal((todo.size, NX, NU)), x
        worst = np.zeros(todo.size)
        for t in range(int(T.max())):
            x = np.einsum("kij,kj->ki", a, x)
            worst = np.where(t < T[todo], np.maximum(worst, np.abs(x).max(1)), worst)
        todo = todo[worst > 5.0]
    n, m = NX * (T + 1) + NU * T, NX * (T + 1)
    xoff = np.cumsum(n) - n
    Td, xo = torch.from_numpy(T).to(DEV), torch.from_numpy(xoff).to(DEV)
    inst = torch.repeat_interleave(torch.arange(count, device=DEV), Td + 1)     # one entry per (problem, step)
    first = torch.cumsum(Td + 1, 0) - (Td + 1)
    t = torch.arange(inst.numel(), device=DEV) - first[inst]                    # 0: the initial state's rows
    i = torch.arange(NX, device=DEV)
    col = torch.empty(inst.numel(), NX, NX + 1 + NU, dtype=torch.int64, device=DEV)
    col[:, :, :NX] = (xo[inst] + NX * (t - 1))[:, None, None] + i[None, None, :]
    col[:, :, NX] = (xo[inst] + NX * t)[:, None] + i[None, :]
    col[:, :, NX + 1:] = (xo[inst] + NX * (Td[inst] + 1) + NU * (t - 1))[:, None, None] + torch.arange(NU, device=DEV)
    val = torch.empty(col.shape, dtype=F64, device=DEV)
    val[:, :, :NX] = -torch.from_numpy(Ad).to(DEV)[inst]
    val[:, :, NX] = 1.0
    val[:, :, NX + 1:] = -torch.from_numpy(Bd).to(DEV)[inst]
    keep = (t > 0)[:, None, None].expand_as(col).clone()
    keep[:, :, NX] = True
    lens = keep.sum(2).reshape(-1)
    N, M = int(n.sum()), int(m.sum())
    Arp = torch.zeros(M + 1, dtype=torch.int64, device=DEV)
    Arp[1:] = torch.cumsum(lens, 0)
    b = torch.zeros(inst.numel(), NX, dtype=F64, device=DEV)
    b[t == 0] = torch.from_numpy(x0).to(DEV)
    u = torch.full((N,), 5.0, dtype=F64, device=DEV)
    nd = torch.from_numpy(n).to(DEV)
    var = torch.arange(N, device=DEV)
    owner = torch.repeat_interleave(torch.arange(count, device=DEV), nd)
    u[var - xo[owner] >= NX * (Td[owner] + 1)] = 1.0
    q = torch.from_numpy(rng.uniform(0.1, 1.0, N)).to(DEV)
    return dict(n=n, m=m, m_eq=m, Q=(torch.arange(N + 1, device=DEV, dtype=I32), var.to(I32), q),
                A=(Arp.to(I32), col[keep].to(I32), val[keep]), c=torch.zeros(N, dtype=F64, device=DEV),
                b=b.reshape(-1), l=-u, u=u)


def _portfolio_qp(seed, n, r):
    """Q = diag + F F'; a budget row and a return row over every asset; 0 <= x <= u."""
    g = _gen(seed, 4)
    A = (torch.tensor([0, n, 2 * n], device=DEV, dtype=I32),
         torch.arange(n, device=DEV, dtype=I32).repeat(2),
         torch.cat([torch.ones(n, dtype=F64, device=DEV), 0.05 + 0.02 * _normal(g, n)]))
    Q = (torch.arange(n + 1, device=DEV, dtype=I32), torch.arange(n, device=DEV, dtype=I32), _uniform(g, 0.01, 0.1, n))
    l, u = _box(n, 0.0, 0.05)
    return dict(n=n, m=2, m_eq=1, Q=Q, A=A, c=torch.zeros(n, dtype=F64, device=DEV),
                b=torch.tensor([1.0, 0.05], dtype=F64, device=DEV), l=l, u=u, F=(0.05 * _normal(g, n, r)).float())


def _arrays(p):
    return (*p["Q"], *p["A"], p["c"], p["b"], p["l"], p["u"])


class _Handle:
    """Keeps a library handle for as long as the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


# --------------------------------------------------------------------------
# the warm-start network
# --------------------------------------------------------------------------
def _family_data(seed, n, m, count, targets):
    """(C, B) around a mean objective and right-hand side, and solver-like outputs near a mean solution."""
    g = _gen(seed, 5)
    out = []
    for k in (n, m):
        out.append(_normal(g, k) + 0.1 * _normal(g, count, k))
    if targets:
        for k, v in ((n, out[0]), (m, out[1])):
            w = _normal(g, k)
            out.append(torch.clamp(w - 0.3 * torch.roll(v, 1, 1) * w - 0.2 * v, -10.0, 10.0))
    return out


def _network(case, seed, data):
    """The network with random weights and the normalisation of `data` (its mean and deviation)."""
    n, m, d = case["n"], case["m"], case["width"]
    g = _gen(seed, 6)
    F = n + m
    w = pdqp.pdqp_ws_create(n, m, d, d, case["depth"], case.get("batch", 512))
    P = (_normal(g, d, F) / math.sqrt(F)).float()
    layers = [((_normal(g, d, d) * math.sqrt(2.0 / d)).float(), 0.1 * _normal(g, d).float()) for _ in range(case["depth"])]
    layers.append(((_normal(g, F, d) * math.sqrt(0.01 / d)).float(), 0.01 * _normal(g, F).float()))
    torch.cuda.synchronize()
    pdqp.pdqp_ws_set_params(w, -1, P)
    for k, (W, b) in enumerate(layers):
        pdqp.pdqp_ws_set_params(w, k, W, b)
    v = torch.cat(data[:2], 1)
    t = torch.cat(data[2:], 1) if len(data) > 2 else v
    std = lambda a: torch.sqrt(((a - a.mean(0)) ** 2).mean(0)) + 1e-3
    norm = [v.mean(0).float(), (1.0 / std(v)).float(), t.mean(0).float(), std(t).float(), (1.0 / std(t)).float()]
    torch.cuda.synchronize()
    pdqp.pdqp_ws_set_normalization(w, *norm)
    return _Handle(w, pdqp.pdqp_ws_destroy), P, layers, norm


# --------------------------------------------------------------------------
# prepare / run
# --------------------------------------------------------------------------
def _problem(case, seed):
    kind = case["kind"]
    if kind == "large":
        return _large_qp(seed, case["n"], case["m"])
    if kind == "portfolio":
        return _portfolio_qp(seed, case["n"], case["r"])
    if kind == "kkt":
        return _control_qps(seed, 1, case["horizon"], case["horizon"])
    if kind == "batch":
        return _control_qps(seed, case["count"], case["t_lo"], case["t_hi"])
    return _gram_qp(seed, case["n"], case["m"], case.get("q_per_row", 5), case.get("a_per_row", 10))


def _options(case):
    mixed = case["precision"] == "mixed"
    return pdqp.pdqp_default_options(precision=pdqp.PDQP_PREC_MIXED if mixed else pdqp.PDQP_PREC_FP64)


def prepare(case, seed):
    kind, st = case["kind"], dict(case=case)
    if kind in ("qp", "large", "batch", "family", "portfolio"):
        p = _problem(case, seed)
        count = case.get("count", 1)
        st["opt"] = _options(case)
        if kind == "batch":
            st["p"] = p
            N, M = int(p["n"].sum()), int(p["m"].sum())
        elif kind == "family":
            g = _gen(seed, 7)
            C, B = p["c"] + 0.1 * _normal(g, count, p["n"]), p["b"] + 0.1 * _normal(g, count, p["m"])
            torch.cuda.synchronize()
            h = pdqp.pdqp_create_family(count, p["n"], p["m"], p["m_eq"], *p["Q"], *p["A"], C, B, p["l"], p["u"])
            N, M = count * p["n"], count * p["m"]
            st["h"] = _Handle(h, pdqp.pdqp_destroy)
        else:
            torch.cuda.synchronize()
            h = pdqp.pdqp_create(p["n"], p["m"], p["m_eq"], *_arrays(p))
            if "F" in p:
                pdqp.pdqp_set_lowrank_Q(h, case["r"], p["F"])
            N, M = p["n"], p["m"]
            st["h"] = _Handle(h, pdqp.pdqp_destroy)
        st["x"], st["y"] = torch.zeros(N, dtype=F64, device=DEV), torch.zeros(M, dtype=F64, device=DEV)
    elif kind == "kkt":
        p = _problem(case, seed)
        n, m = int(p["n"][0]), int(p["m"][0])
        rp, col, val = p["A"]
        row = torch.repeat_interleave(torch.arange(m, device=DEV), (rp[1:] - rp[:-1]).long())
        g = _gen(seed, 8)
        x = torch.minimum(torch.maximum(0.5 * _normal(g, n), p["l"]), p["u"])
        st["args"] = (n, m, m, *p["Q"], *p["A"], *_csr(col.long(), row, val, n, m), p["c"], p["b"], p["l"], p["u"], x,
                      0.1 * _normal(g, m), torch.zeros(6, dtype=F64, device=DEV))
    elif kind == "fit":
        st["data"] = _family_data(seed, case["n"], case["m"], case["count"], True)
        torch.cuda.synchronize()
        st["w"] = _Handle(pdqp.pdqp_ws_create(case["n"], case["m"], 64, 64, 1, 64), pdqp.pdqp_ws_destroy)
    elif kind in ("train", "infer"):
        st["data"] = _family_data(seed, case["n"], case["m"], case["count"], kind == "train")
        st["w"], _, layers, _ = _network(case, seed, st["data"])
        if kind == "train":
            st["layers"] = [(torch.empty_like(W), torch.empty_like(b)) for W, b in layers]
        else:
            st["out"] = [torch.zeros(case["count"], k, dtype=F64, device=DEV) for k in (case["n"], case["m"])]
    else:
        g = _gen(seed, 9)
        M, N, K = case["M"], case["N"], case["K"]
        st["A"], st["B"] = (torch.randn(k, K, generator=g, device=DEV).bfloat16() for k in (M, N))
        if case["epilogue"] == "plain":
            st["kw"] = dict(D_f32=torch.zeros(M, N, device=DEV))
        else:
            st["kw"] = dict(D_bf16=torch.zeros(M, N, device=DEV, dtype=torch.bfloat16), relu=True,
                            bias=torch.randn(N, generator=g, device=DEV))
        splits = pdqp.pdqp_gemm_bf16_splits(M, N, K, 0)
        if splits > 1:
            st["kw"]["workspace"] = torch.empty(splits * M * N, device=DEV)
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        p = st["p"]
        h = pdqp.pdqp_create_batch_packed(p["n"], p["m"], p["m_eq"], *_arrays(p))
        status, info = pdqp.pdqp_solve(h, st["opt"], x_out=st["x"], y_out=st["y"])
        pdqp.pdqp_destroy(h)
        return dict(status=status, x=st["x"], y=st["y"])
    if kind in ("qp", "large", "family", "portfolio"):
        status, info = pdqp.pdqp_solve(st["h"].h, st["opt"], x_out=st["x"], y_out=st["y"])
        return dict(status=status, objective=info.primal_obj, x=st["x"], y=st["y"])
    if kind == "kkt":
        pdqp.pdqp_kkt_noalloc(*st["args"], stream=torch.cuda.current_stream())
        return st["args"][-1]
    if kind == "fit":
        w, F = st["w"].h, case["n"] + case["m"]
        pdqp.pdqp_ws_fit(w, *st["data"])
        return pdqp.pdqp_ws_get_normalization(w, F)
    if kind == "train":
        losses = pdqp.pdqp_ws_train(st["w"].h, *st["data"], epochs=1, batch=case["batch"], lr=1e-4, seed=1)
        for k, (W, b) in enumerate(st["layers"]):
            pdqp.pdqp_ws_get_params(st["w"].h, k, 0, W, b)
        return dict(losses=losses, layers=st["layers"])
    if kind == "infer":
        pdqp.pdqp_ws_infer(st["w"].h, *st["data"], *st["out"])
        return st["out"]
    pdqp.pdqp_gemm_bf16(st["A"], st["B"], stream=torch.cuda.current_stream(), **st["kw"])
    return st["kw"].get("D_f32", st["kw"].get("D_bf16"))


# --------------------------------------------------------------------------
# work / exact
# --------------------------------------------------------------------------
def work(case):
    """Bytes: each input read once, each output written once (a solve's iterations may keep what they
    read on the chip).  Flops: those of one product with each matrix; of the network, its GEMMs."""
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=2 * (M * K + N * K) + (4 if case["epilogue"] == "plain" else 2) * M * N, flops=2 * M * N * K)
    if kind in ("fit", "train", "infer"):
        F, count = case["n"] + case["m"], case["count"]
        if kind == "fit":
            return dict(bytes=16 * count * F + 20 * F, flops=10 * count * F)
        w, depth = case["width"], case["depth"]
        weights = depth * w * w + F * w
        forward = 2 * count * (F * w + weights)
        if kind == "infer":
            return dict(bytes=16 * count * F + 2 * (weights + F * w), flops=forward)
        steps = count // case["batch"]
        return dict(bytes=16 * count * F + 2 * F * w + steps * 24 * weights, flops=forward + 2 * 2 * count * weights)
    count = case.get("count", 1)
    if kind in ("batch", "kkt"):
        T = case["horizon"] if kind == "kkt" else (case["t_lo"] + case["t_hi"]) / 2
        n, m = NX * (T + 1) + NU * T, NX * (T + 1)
        nnz_Q, nnz_A = n, NX + NX * (NX + 1 + NU) * T
    elif kind == "large":
        n, m = case["n"], case["m"]
        nnz_Q, nnz_A = 6 * n, 10 * n
    elif kind == "portfolio":
        n, m = case["n"], 2
        nnz_Q, nnz_A = n, 2 * n
    else:
        n, m = case["n"], case["m"]
        k = case.get("q_per_row", 5)
        nnz_Q, nnz_A = n * (k * (k - 1) + 1), m * case.get("a_per_row", 10)
    F = 4 * n * case.get("r", 0)
    if kind == "family":
        bytes_ = 12 * (nnz_Q + nnz_A) + 16 * n + count * 16 * (n + m)
    elif kind == "kkt":
        bytes_ = 12 * (nnz_Q + 2 * nnz_A) + 4 * (2 * n + m) + 8 * (4 * n + 2 * m) + 48
    else:
        bytes_ = count * (12 * (nnz_Q + nnz_A) + 4 * (n + m) + 8 * (4 * n + 2 * m) + F)
    return dict(bytes=int(bytes_), flops=int(count * (2 * nnz_Q + 4 * nnz_A + F)))


def _visit(seed, epoch, count):
    """The documented visit order of a training epoch: i -> (a i + s) mod count."""
    mask = (1 << 64) - 1

    def mix(z):
        z = (z + 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    z = mix((seed * 0x9E3779B97F4A7C15 + epoch * 0xD1B54A32D192ED03) & mask)
    a = (z % count) | 1
    while math.gcd(a, count) != 1:
        a += 2
    a %= count
    return (a or 1), (z >> 32) % count


def _exact_train(case, seed):
    data = _family_data(seed, case["n"], case["m"], case["count"], True)
    _, P, layers, (im, isc, om, _, oi) = _network(case, seed, data)
    H0 = ((torch.cat(data[:2], 1) - im.double()) * isc.double()) @ P.double().T
    T = (torch.cat(data[2:], 1) - om.double()) * oi.double()
    params = [t.double() for layer in layers for t in layer]
    m1, m2 = [torch.zeros_like(t) for t in params], [torch.zeros_like(t) for t in params]
    batch, count = case["batch"], case["count"]
    a, s = _visit(1, 0, count)
    loss, steps = 0.0, count // batch
    for k in range(steps):
        idx = (a * torch.arange(k * batch, (k + 1) * batch, device=DEV) + s) % count
        hs = [H0[idx]]
        for j in range(case["depth"]):
            hs.append(torch.relu(hs[-1] @ params[2 * j].T + params[2 * j + 1]))
        d = hs[-1] @ params[-2].T + params[-1] - T[idx]
        loss += float((d * d).mean())
        g = 2.0 * d / d.numel()
        grads = [None] * len(params)
        for j in range(case["depth"], -1, -1):
            grads[2 * j], grads[2 * j + 1] = g.T @ hs[j], g.sum(0)
            if j:
                g = (g @ params[2 * j]) * (hs[j] > 0)
        for i, gr in enumerate(grads):
            m1[i].mul_(0.9).add_(gr, alpha=0.1)
            m2[i].mul_(0.999).addcmul_(gr, gr, value=0.001)
            params[i] -= 1e-4 * (m1[i] / (1 - 0.9 ** (k + 1))) / (torch.sqrt(m2[i] / (1 - 0.999 ** (k + 1))) + 1e-8)
    return dict(losses=np.array([loss / steps]), layers=[(params[2 * j], params[2 * j + 1]) for j in range(len(layers))])


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        st = prepare(case, seed)
        d = st["A"].double() @ st["B"].double().T
        return d if case["epilogue"] == "plain" else torch.relu(d + st["kw"]["bias"].double())
    if kind == "kkt":
        n, m, m_eq, qr, qc, qv, ar, ac, av, tr, tc, tv, c, b, l, u, x, y, _ = prepare(case, seed)["args"]
        Qx, Ax, ATy = _row_sums((qr, qc, qv), x), _row_sums((ar, ac, av), x), _row_sums((tr, tc, tv), y)
        g = Qx + c - ATy
        lf, uf = torch.isfinite(l), torch.isfinite(u)
        zero = torch.zeros_like(g)
        lam = torch.where(lf & uf, g, torch.where(lf, g.clamp(min=0), torch.where(uf, g.clamp(max=0), zero)))
        viol = Ax - b
        viol[m_eq:] = (-viol[m_eq:]).clamp(min=0)
        top = lambda *v: max(float(t.abs().max()) for t in v)
        box = torch.where(lam > 0, l * lam, torch.where(lam < 0, u * lam, zero)).sum()
        pobj = float(0.5 * (x @ Qx) + c @ x)
        dobj = float(-0.5 * (x @ Qx) + b @ y + box)
        rp, rd = top(viol) / (1 + top(Ax, b)), top(g - lam) / (1 + top(Qx, ATy, c))
        rg = abs(pobj - dobj) / (1 + max(abs(pobj), abs(dobj)))
        return torch.tensor([rp, rd, rg, max(rp, rd, rg), pobj, dobj], dtype=F64)
    if kind == "fit":
        C, B, X, Y = _family_data(seed, case["n"], case["m"], case["count"], True)
        mean = lambda *v: torch.cat([a.mean(0) for a in v])
        std = lambda *v: torch.cat([torch.sqrt(((a - a.mean(0)) ** 2).mean(0)) for a in v])
        fix = lambda s: torch.where(s < 1e-8, torch.ones_like(s), s)
        s_in, s_out = fix(std(C, B)), fix(std(X, Y))
        return dict(in_mean=mean(C, B), in_scale=1 / s_in, out_mean=mean(X, Y), out_std=s_out, out_inv=1 / s_out)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "infer":
        data = _family_data(seed, case["n"], case["m"], case["count"], False)
        _, P, layers, (im, isc, om, os_, _) = _network(case, seed, data)
        h = ((torch.cat(data, 1) - im.double()) * isc.double()) @ P.double().T
        for W, b in layers[:-1]:
            h = torch.relu(h @ W.double().T + b.double())
        o = om.double() + os_.double() * (h @ layers[-1][0].double().T + layers[-1][1].double())
        return [o[:, :case["n"]].contiguous(), o[:, case["n"]:].contiguous()]
    return None     # a solve's answer is one of many points within its tolerance
