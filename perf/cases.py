"""The work that users of the library have it do, as cases that can be timed.

Every case goes through the package's public entry points. Inputs are the
synthetic workloads of the package's generators (Gaussian mixtures, 8-bit
sparse prototypes, Gamma and log-normal clusters), drawn on the GPU.

kind            what it stands for
p               a data set's similarity matrix: exact kNN, beta bisection, CSR P
forest          the approximate neighbourhoods of a data set: forest build and search
forest_rows     points inserted by a forest search of a resident forest
refine          exact neighbourhoods of the rows under the lens, written back
refine_batch    many brushed selections refined in one call
insert          a batch of points inserted exactly into a served state
csr             the resident CSR P rebuilt after commits: bisection and symmetrisation
view            the density, selection and approximation maps of an embedding
"""
import math

import torch

import paper_1512_01655_gb300 as at

DEV = "cuda"


def listed():
    return [
        # the small data set of the parity workload: launches and latency count
        dict(name="p_gaussian_2k_x64", kind="p", data="gaussian", N=2000, D=64, perplexity=30.0, precision="fp32"),
        # an MNIST-shaped data set, 8-bit values, in the default mode
        dict(name="p_bytes_70k_x784", kind="p", data="bytes", N=70000, D=784, perplexity=30.0, precision="fp32"),
        # an ordinary data set of odd sizes at the largest usual perplexity (k = 150)
        dict(name="p_lognormal_50021_x50", kind="p", data="lognormal", N=50021, D=50, perplexity=50.0,
             precision="fp32"),
        # the headline workload: BF16 distances, the top 4k re-ranked
        dict(name="p_gamma_1m_x128_bf16", kind="p", data="gamma", N=1000000, D=128, perplexity=30.0,
             precision="bf16_approx"),
        # the same features in the default mode (three passes, certified exact)
        dict(name="p_gamma_200k_x128", kind="p", data="gamma", N=200000, D=128, perplexity=30.0, precision="fp32"),
        # the paper's approximate neighbourhoods of the MNIST-shaped set
        dict(name="forest_bytes_70k_x784", kind="forest", data="bytes", N=70000, D=784, k=90, trees=4, checks=1024),
        # an insertion into a served corpus takes its neighbourhoods from the resident forest
        dict(name="forest_rows_5k_of_200k", kind="forest_rows", data="lognormal", N=200000, D=50, S=5000, k=90,
             trees=4, checks=1024),
        # a lens over a few hundred points of the MNIST-shaped set
        dict(name="refine_500_of_70k_x784", kind="refine", data="bytes", N=70000, D=784, S=500, perplexity=30.0),
        # brushed selections of a large corpus
        dict(name="refine_batch_64_of_500k", kind="refine_batch", data="gaussian", N=500000, D=256, subsets=64,
             lo=200, hi=20000, perplexity=30.0),
        # a served corpus takes a batch of new points exactly
        dict(name="insert_7013_into_100k", kind="insert", data="lognormal", N=100000, D=50, B=7013,
             perplexity=30.0),
        # the served CSR P after commits
        dict(name="csr_300k_k90", kind="csr", N=300000, perplexity=30.0),
        # the view of the MNIST-shaped set's embedding
        dict(name="view_70k_1024px", kind="view", N=70000, width=1024, height=1024, h=0.3, cutoff=4.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["p", "p", "p", "forest", "forest_rows", "refine", "refine_batch", "insert", "csr", "view"])
    perp = rng.choice([10.0, 20.0, 30.0, 30.0, 50.0])
    if kind in ("refine", "refine_batch"):
        perp = min(perp, 30.0)
    k = int(3 * perp)
    if kind == "p":
        data = rng.choice(["gaussian", "bytes", "lognormal", "gamma"])
        D = _log_int(rng, 16, 784)
        if data == "gamma":
            precision = rng.choice(["fp32", "bf16_approx", "bf16_approx", "fp8"])
        else:
            precision = rng.choice(["fp32", "bf16"]) if data == "bytes" else "fp32"
        N = _log_int(rng, 1000, 1000000 if precision in ("bf16_approx", "fp8") else 200000)
        passes = 3 if precision == "fp32" else 1
        while float(N) * N * (D * passes + 200) > 3e14:
            N = N * 3 // 4
        return dict(kind=kind, data=data, N=N, D=D, perplexity=perp, precision=precision)
    if kind == "forest":
        return dict(kind=kind, data=rng.choice(["bytes", "bytes", "lognormal", "gaussian"]),
                    N=_log_int(rng, 2000, 150000), D=_log_int(rng, 16, 784), k=min(k, 90),
                    trees=rng.choice([2, 4, 8]), checks=rng.choice([256, 512, 1024]))
    if kind == "forest_rows":
        N = _log_int(rng, 20000, 400000)
        return dict(kind=kind, data=rng.choice(["lognormal", "gaussian"]), N=N, D=_log_int(rng, 16, 256),
                    S=_log_int(rng, 500, min(20000, N // 4)), k=min(k, 90), trees=rng.choice([2, 4]),
                    checks=rng.choice([256, 1024]))
    if kind == "refine":
        N = _log_int(rng, 10000, 300000)
        return dict(kind=kind, data=rng.choice(["bytes", "lognormal", "gaussian"]), N=N, D=_log_int(rng, 32, 784),
                    S=_log_int(rng, 200, min(20000, N // 4)), perplexity=perp)
    if kind == "refine_batch":
        return dict(kind=kind, data="gaussian", N=_log_int(rng, 50000, 500000), D=_log_int(rng, 32, 256),
                    subsets=rng.randint(8, 64), lo=200, hi=rng.choice([2000, 5000, 20000]), perplexity=perp)
    if kind == "insert":
        N = _log_int(rng, 20000, 400000)
        return dict(kind=kind, data=rng.choice(["lognormal", "gaussian"]), N=N, D=_log_int(rng, 16, 128),
                    B=_log_int(rng, 1000, 20000), perplexity=perp)
    if kind == "csr":
        return dict(kind=kind, N=_log_int(rng, 5000, 1000000), perplexity=perp)
    return dict(kind=kind, N=_log_int(rng, 5000, 200000), width=rng.randint(300, 1200), height=rng.randint(300, 1200),
                h=rng.choice([0.1, 0.3, 0.5]), cutoff=rng.choice([3.0, 4.0]))


# ---- inputs -------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rows(data, N, D, g):
    """(X float32 [N][D], cluster of each row)"""
    def uni(*shape):
        return torch.rand(shape, generator=g, device=DEV)

    def nrm(*shape):
        return torch.randn(shape, generator=g, device=DEV)

    M = {"gaussian": 100 if N >= 50000 else 10, "bytes": 10, "lognormal": 30, "gamma": 50}[data]
    lab = torch.randint(M, (N,), generator=g, device=DEV)
    if data == "gaussian":
        X = (4.0 * nrm(M, D))[lab] + nrm(N, D)
    elif data == "lognormal":
        X = torch.exp(nrm(M, D)[lab] + nrm(N, D))
    elif data == "gamma":  # Gamma(2, 1): the sum of two exponentials
        e = -torch.log(uni(N, D).clamp_(min=1e-30)) - torch.log(uni(N, D).clamp_(min=1e-30))
        X = (0.5 + 1.5 * uni(M, D))[lab] * e
    else:
        val, sup = 64.0 + 191.0 * uni(M, D), uni(M, D) < 0.2
        on = (sup[lab] & (uni(N, D) < 0.95)) | (uni(N, D) < 0.02)
        X = torch.where(on, (val[lab] + 40.0 * nrm(N, D)).round().clamp(0, 255), torch.zeros((), device=DEV))
    return X.contiguous(), lab


def _pick(N, S, g):
    return torch.randperm(N, generator=g, device=DEV)[:S].sort().values.to(torch.int32)


def _approximate(X, k, perp):
    """The approximate neighbourhoods and conditionals a program holds before it refines."""
    f = at.atsne_forest_build(X, trees=4, checks=k, leaf_size=1, seed=7)
    idx, d2, _ = at.atsne_forest_query(X, f, k)
    P, beta = at.atsne_calibrate_P(d2, perp)
    return idx, d2, P, beta


def _cluster_lists(N, k, g):
    """kNN lists of log-normal points in separate clusters, rows shuffled: the
    neighbours of a row lie in its own cluster, scattered over the corpus."""
    m = 1000 if N >= 4000 else max(k + 1, N // 4)
    idx = torch.empty((N, k), dtype=torch.int32, device=DEV)
    d2 = torch.empty((N, k), dtype=torch.float32, device=DEV)
    perm = torch.randperm(N, generator=g, device=DEV)
    for s in range(0, N, m):
        n = min(m, N - s)
        if n <= k:  # a short last cluster joins the rows before it
            s, n = N - m, m
        X = torch.exp(torch.randn((n, 24), generator=g, device=DEV))
        D2 = torch.cdist(X, X).square_()
        D2.fill_diagonal_(math.inf)
        d, j = D2.topk(k, largest=False)
        r = perm[s:s + n]
        idx[r], d2[r] = r[j].to(torch.int32), d
    return idx, d2


def _csr_buffers(N, k):
    """Buffers for the CSR P of any lists (at most 2Nk entries; the rest stays 0)."""
    return (torch.zeros(N + 1, dtype=torch.int64, device=DEV), torch.zeros(2 * N * k, dtype=torch.int32, device=DEV),
            torch.zeros(2 * N * k, dtype=torch.float32, device=DEV), torch.zeros(1, dtype=torch.int64, device=DEV))


def prepare(case, seed):
    g, c, kind = _gen(seed), case, case["kind"]
    if kind == "csr":
        k = int(3 * c["perplexity"])
        idx, d2 = _cluster_lists(c["N"], k, g)
        ws = torch.empty(at.workspace_bytes(at.OP_SYMMETRIZE, c["N"], 0, k), dtype=torch.uint8, device=DEV)
        return dict(case=c, idx=idx, d2=d2, P=torch.empty_like(d2), out=_csr_buffers(c["N"], k), ws=ws)
    if kind == "view":
        lab = torch.randint(10, (c["N"],), generator=g, device=DEV)
        ang = lab * (2 * math.pi / 10)
        Y = torch.stack([10 * ang.cos(), 10 * ang.sin()], 1)
        Y = Y + (0.5 + torch.rand((10, 2), generator=g, device=DEV))[lab] * \
            torch.randn((c["N"], 2), generator=g, device=DEV)
        rho = torch.rand(c["N"], generator=g, device=DEV)
        lo = Y.amin(0) - 1
        pixel = float(((Y.amax(0) + 1 - lo) / torch.tensor([c["width"], c["height"]], device=DEV)).max())
        return dict(case=c, Y=Y.contiguous(), rho=rho, sel=(lab == 3).to(torch.uint8), x0=float(lo[0]),
                    y0=float(lo[1]), pixel=pixel)
    X, lab = _rows(c["data"], c["N"] + c.get("B", 0), c["D"], g)
    s = dict(case=c, X=X)
    if kind == "p":
        s["out"] = _csr_buffers(c["N"], int(3 * c["perplexity"]))
    elif kind == "forest_rows":
        s["forest"] = at.atsne_forest_build(X, trees=c["trees"], checks=c["checks"], leaf_size=1, seed=7)
        s["rows"] = _pick(c["N"], c["S"], g)
    elif kind == "refine":
        s["rows"] = _pick(c["N"], c["S"], g)
        s["lists"] = _approximate(X, int(3 * c["perplexity"]), c["perplexity"])
        s["hint"] = s["lists"][1][:, -1][s["rows"].long()].contiguous()
        s["rho"] = torch.zeros(c["N"], device=DEV)
    elif kind == "refine_batch":
        # each selection: log-uniform size, members from one to three clusters
        r = torch.rand((c["subsets"],), generator=g, device=DEV).tolist()
        members = []
        for u in r:
            size = int(math.exp(math.log(c["lo"]) + u * math.log(c["hi"] / c["lo"])))
            cl = torch.randint(int(lab.max()) + 1, (3,), generator=g, device=DEV)
            pool = (lab.unsqueeze(1) == cl[:1 + size % 3]).any(1).nonzero().flatten()
            members.append(pool[torch.randperm(pool.numel(), generator=g, device=DEV)[:size]].sort().values)
        s["sel"] = torch.cat(members).to(torch.int32)
        s["lists"] = _approximate(X, int(3 * c["perplexity"]), c["perplexity"])
        s["state"] = [t.clone() for t in s["lists"]] + [torch.zeros(c["N"], device=DEV)]
    elif kind == "insert":
        k = int(3 * c["perplexity"])
        s["idx"], s["d2"] = at.atsne_knn(X[:c["N"]], k)
        s["rows"] = torch.arange(c["N"], c["N"] + c["B"], dtype=torch.int32, device=DEV)
    return s


# ---- one pass -----------------------------------------------------------------

def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "p":
        idx, d2 = at.atsne_knn(s["X"], int(3 * c["perplexity"]), precision=c["precision"])
        P, beta = at.atsne_calibrate_P(d2, c["perplexity"])
        return [idx, d2, P, beta, *at.atsne_symmetrize(idx, P, trim=False, out=s["out"])]
    if kind == "forest":
        return list(at.atsne_knn(s["X"], c["k"], method="forest", trees=c["trees"], checks=c["checks"], seed=7))
    if kind == "forest_rows":
        return list(at.atsne_forest_query(s["X"], s["forest"], c["k"], queries=s["rows"]))
    if kind == "refine":
        # as the serving loop refines: search, bisection, the rows written back
        idx, d2, P, beta = s["lists"]
        ti, td = at.atsne_knn_rows(s["X"], s["rows"], idx.shape[1], hint_d2=s["hint"])
        tp, tb = at.atsne_calibrate_P(td, c["perplexity"])
        at.atsne_commit_rows(s["rows"], ti, td, tp, tb, idx, d2, P, beta, s["rho"])
        return [ti, td, tp, tb, idx, d2, P, beta, s["rho"]]
    if kind == "refine_batch":
        # every pass starts from the approximate neighbourhoods
        for t, t0 in zip(s["state"], s["lists"]):
            t.copy_(t0)
        idx, d2, P, beta, rho = s["state"]
        n = at.atsne_refine_batch(s["X"], s["sel"], c["perplexity"], idx, d2, P, beta, rho)
        return [idx, d2, P, beta, rho, n]
    if kind == "insert":
        # the state before stays as it is: the merge goes into copies
        N, k, X = c["N"], s["idx"].shape[1], s["X"]
        ti, td = at.atsne_knn(X, k, queries=s["rows"])
        tp, tb = at.atsne_calibrate_P(td, c["perplexity"])
        ci, cd = at.atsne_knn_cross(X[:N], X[N:], min(k, c["B"]), radius_d2=at.atsne_row_dmax(s["d2"]))
        idx, d2 = s["idx"].clone(), s["d2"].clone()
        at.atsne_merge_neighbors(idx, d2, ci, cd, N)
        return [ti, td, tp, tb, idx, d2, *at.atsne_calibrate_P(d2, c["perplexity"])]
    if kind == "csr":
        P, beta = at.atsne_calibrate_P(s["d2"], c["perplexity"], P_out=s["P"])
        return [P, beta, *at.atsne_symmetrize(s["idx"], P, trim=False, out=s["out"], workspace=s["ws"])]
    return list(at.atsne_kde_map(s["Y"], s["x0"], s["y0"], s["pixel"], c["width"], c["height"], c["h"],
                                 cutoff=c["cutoff"], rho=s["rho"], selected=s["sel"]))


# ---- the least a pass moves and computes ---------------------------------------

def work(case):
    c, kind = case, case["kind"]
    N, D = c["N"], c.get("D", 0)
    k = c["k"] if "k" in c else int(3 * c.get("perplexity", 0))
    x, lists = 4.0 * N * D, 8.0 * N * k
    steps = 20 * 4.0 * k  # a row's bisection: about twenty sums over its neighbours
    # the joint P holds each of the Nk entries and its transpose, mutual ones once
    csr = 8.0 * (N + 1) + 8.0 * 1.6 * N * k
    if kind == "p":
        return dict(bytes=x + lists + 4.0 * N * k + 4 * N + csr, flops=2.0 * N * N * D + N * steps)
    if kind == "forest":
        # rows read once and the lists written; per query: checks distances
        return dict(bytes=x + lists, flops=2.0 * N * c["checks"] * D)
    if kind == "forest_rows":
        S = c["S"]
        return dict(bytes=min(x, 4.0 * S * c["checks"] * D) + S * (8.0 * k + 8), flops=2.0 * S * c["checks"] * D)
    if kind == "refine":
        S = c["S"]
        return dict(bytes=x + 2 * S * (12.0 * k + 8), flops=2.0 * S * N * D + S * steps)
    if kind == "refine_batch":
        S = min(0.9 * N, c["subsets"] * (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"]))
        return dict(bytes=x + 2 * (12.0 * N * k + 8 * N), flops=2.0 * S * N * D + S * steps)
    if kind == "insert":
        B = c["B"]
        return dict(bytes=x + 4.0 * B * D + 2 * lists + 4.0 * N * k + 12.0 * B * k,
                    flops=2.0 * B * (2 * N + B) * D + (N + B) * steps)
    if kind == "csr":
        return dict(bytes=lists + 4.0 * N * k + 4 * N + csr, flops=N * steps)
    w, h = c["width"], c["height"]
    # each pixel's Gaussians over the points within reach of it (about 6% of an image of ten clusters)
    return dict(bytes=13.0 * N + 16.0 * w * h, flops=8.0 * 0.06 * N * w * h * min(1.0, (c["h"] / 0.3) ** 2))


# ---- the same in 64 bits --------------------------------------------------------

def _knn64(Q, X, k, self_at=None):
    """(idx, d2) of each row of Q among X's, ordered by (d2, index); self_at: each row's own index."""
    Q, X = Q.double(), X.double()
    xx = X.square().sum(1)
    kk = min(k + 6, X.shape[0] - (self_at is not None))
    step = max(1, int(1.5e9 / 8 / X.shape[0]))
    idx, d2 = [], []
    for a in range(0, Q.shape[0], step):
        q = Q[a:a + step]
        K = torch.addmm(xx, q, X.t(), alpha=-2.0)
        if self_at is not None:
            K.scatter_(1, self_at[a:a + step].long().unsqueeze(1), math.inf)
        j = K.topk(kk, largest=False).indices.sort(1).values
        for b in range(0, j.shape[0], 1024):  # the distances themselves as sums of squared differences
            jb = j[b:b + 1024]
            d = torch.zeros(jb.shape, dtype=torch.float64, device=DEV)
            for e in range(0, X.shape[1], 128):
                d += (X[:, e:e + 128][jb] - q[b:b + 1024, None, e:e + 128]).square().sum(2)
            d, o = d.sort(dim=1, stable=True)
            idx.append(jb.gather(1, o)[:, :k])
            d2.append(d[:, :k])
    return torch.cat(idx), torch.cat(d2)


def _bisect64(d2, perp):
    """(P, beta): the bandwidth at which each row's perplexity is the target."""
    s = d2.double()
    s = s - s.amin(1, keepdim=True)
    lo, hi = torch.zeros(s.shape[0], device=DEV).double(), torch.full((s.shape[0],), math.inf, device=DEV).double()
    beta = torch.ones_like(lo)
    for _ in range(100):
        w = torch.exp(-beta[:, None] * s)
        z = w.sum(1)
        up = z.log() + beta * (w * s).sum(1) / z > math.log(perp)
        lo, hi = torch.where(up, beta, lo), torch.where(up, hi, beta)
        beta = torch.where(hi.isinf(), 2 * beta, 0.5 * (lo + hi))
    w = torch.exp(-beta[:, None] * s)
    return w / w.sum(1, keepdim=True), beta


def _joint64(idx, P):
    """The values of the symmetrised P in row order, columns ascending, in a buffer of 2Nk."""
    N, k = idx.shape
    i = torch.arange(N, device=DEV).repeat_interleave(k)
    j = idx.flatten().long()
    key, o = torch.cat([i * N + j, j * N + i]).sort(stable=True)
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    val = torch.zeros(2 * N * k, dtype=torch.float64, device=DEV)
    p = P.double().flatten()
    val.index_add_(0, first.cumsum(0) - 1, torch.cat([p, p])[o])
    return val / (2.0 * N)


def exact(case, seed):
    c, kind = case, case["kind"]
    perp, k = c.get("perplexity"), int(3 * c.get("perplexity", 0))
    if kind in ("forest", "forest_rows", "refine_batch"):
        return None
    if kind in ("csr", "view"):
        s = prepare(c, seed)
        if kind == "view":
            return _view64(s)
        P, beta = _bisect64(s["d2"], perp)
        return [P, beta, None, None, _joint64(s["idx"], P), None]
    N, D = c["N"], c["D"]
    if kind == "p":
        if 2.0 * N * N * D > 1e13 or N > 80000:
            return None
        X = _rows(c["data"], N, D, _gen(seed))[0]
        idx, d2 = _knn64(X, X, k, torch.arange(N, device=DEV))
        P, beta = _bisect64(d2, perp)
        return [None, d2, P, beta, None, None, _joint64(idx, P), None]
    if kind == "refine":
        if 2.0 * c["S"] * N * D > 1e13:
            return None
        g = _gen(seed)
        X = _rows(c["data"], N, D, g)[0]
        rows = _pick(N, c["S"], g)
        _, d2 = _knn64(X[rows.long()], X, k, rows)
        P, beta = _bisect64(d2, perp)
        return [None, d2, P, beta, None, None, None, None, None]
    B = c["B"]
    if float(N + B) * (N + B) > 1.3e10:
        return None
    X = _rows(c["data"], N + B, D, _gen(seed))[0]
    # the state holds exact lists, so the merged ones are exact lists of the grown corpus
    _, d2 = _knn64(X, X, k, torch.arange(N + B, device=DEV))
    P, beta = _bisect64(d2, perp)
    return [None, d2[N:], P[N:], beta[N:], None, d2[:N], P[:N], beta[:N]]


def _view64(s):
    # pixel centres, and which points lie within the cutoff, in 32 bits as the interface states; the sums in 64
    def f32(t):
        return t.float().double()

    c = s["case"]
    Y, rho, sel = s["Y"].double(), s["rho"].double(), s["sel"].double()
    h, px, x0, y0 = (float(t) for t in torch.tensor([c["h"], s["pixel"], s["x0"], s["y0"]]))
    r = float(torch.tensor(float(torch.tensor(c["cutoff"])) * h))
    cx = f32(x0 + (torch.arange(c["width"], device=DEV).double() + 0.5) * px)
    cy = f32(y0 + (torch.arange(c["height"], device=DEV).double() + 0.5) * px)
    F, S, R = (torch.zeros((c["height"], c["width"]), dtype=torch.float64, device=DEV) for _ in range(3))
    for i in range(c["height"]):
        near = ((Y[:, 1] - cy[i]).abs() <= r * 1.001).nonzero().flatten()
        dx, dy = f32(cx[:, None] - Y[near, 0]), f32(cy[i] - Y[near, 1])
        d2 = f32(dx.square() + f32(dy.square()))
        g = torch.where(d2 <= float(torch.tensor(r * r)), torch.exp(-d2 / (2 * h * h)), 0.0) / (2 * math.pi * h * h)
        F[i], S[i], R[i] = g.sum(1), g @ sel[near], g @ rho[near]
    some = F > 0
    a = torch.where(some, R / F, 1.0)
    return [F / c["N"], torch.where(some, S / F, 0.0), a, 1 - a.square()]
