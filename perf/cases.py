"""The work that programs have this library do, as cases that can be timed.

Five kinds of pass, each through the public entry points:

* ``mttkrp``  spMTTKRP along every mode on a plan that the program keeps (the
              inner loop of any CP method that brings its own update);
* ``als``     a CP-ALS run of a few sweeps from given starting factors on a
              kept plan (a restart, or one more starting point);
* ``batch``   the same for many tensors at once, in shared launches;
* ``plan``    the mode copies and partitions of a new tensor;
* ``serve``   jobs submitted to a server and stepped until all are done.

Tensors are drawn on the device: each coordinate uniform or truncated Zipf,
repeated cells dropped, in random order; values U(0,1) or lognormal; factors
N(0,1).  Factors are FP32 or BF16; a decomposition's weights come back in the
factors' type, as a stored model keeps them, its fit in FP32.
"""
import math

import numpy as np
import torch

import paper_2503_18198_gb300 as spm

NNZ_PER_PARTITION = 131072  # partition size of batched and served tensors


# ---- the cases ---------------------------------------------------------------

def _case(name, kind, dims, nnz, rank, dtype="fp32", alphas="", values="uniform", sweeps=0):
    return {"name": name, "kind": kind, "dims": dims, "alphas": alphas, "nnz": nnz, "rank": rank,
            "dtype": dtype, "values": values, "sweeps": sweeps}


def listed():
    return [
        # the smallest tensor in use: latency and launches are all there is
        _case("mttkrp plain", "mttkrp", "64x48x32", 4096, 16),
        # one mid-sized member of a collection of small tensors, BF16 factors
        _case("mttkrp member bf16", "mttkrp", "4000x1500x700", 300_000, 32, "bf16"),
        # a rank that is no power of two, sizes that divide by nothing
        _case("mttkrp rank 24", "mttkrp", "30011x20003x4001", 2_000_003, 24, alphas="1.1,1.1,1.1"),
        # a large skewed tensor with far more rows than fit in cache: the headline workload
        _case("mttkrp scale", "mttkrp", "1000000x500000x200000", 50_000_000, 32,
              alphas="1.2,1.2,1.2"),
        # four modes, one of them short, wide BF16 rows, heavy-tailed values
        _case("mttkrp four modes bf16", "mttkrp", "20000x20000x5000x24", 30_000_000, 64, "bf16",
              "1.0,1.0,1.0,", "lognormal"),
        # the smallest decomposition: a sweep is a chain of tiny launches
        _case("als plain", "als", "64x48x32", 4096, 16, sweeps=3),
        # one request of a decomposition service: four modes, rank 64, BF16 factors
        _case("als request bf16", "als", "30000x8000x2000x300", 3_000_000, 64, "bf16",
              "1.1,1.1,1.1,1.1", sweeps=2),
        # a large decomposition: long factors, so the row updates count as much as the MTTKRP
        _case("als scale", "als", "1000000x500000x200000", 20_000_000, 32, alphas="1.2,1.2,1.2",
              sweeps=3),
        # many independent small tensors decomposed together
        {"name": "batch bf16", "kind": "batch", "count": 96, "nnz": 2_000_000, "dtype": "bf16",
         "sweeps": 2},
        # a new small tensor: what stands before its first sweep
        _case("plan small", "plan", "400x250x120", 30_000, 16, alphas="1.1,1.1,1.1"),
        # a new large tensor
        _case("plan scale", "plan", "1000000x500000x200000", 50_000_000, 32, alphas="1.2,1.2,1.2"),
        # a queue of decomposition jobs of 3 and 4 modes and ranks 8 to 64, start to finish
        {"name": "serve bf16", "kind": "serve", "count": 10, "nnz": 3_000_000, "dtype": "bf16",
         "sweeps": 2},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["mttkrp", "mttkrp", "als", "als", "plan", "batch", "serve"])
    dtype = rng.choice(["fp32", "bf16"])
    # early sweeps move the factors most; rounding to BF16 makes later ones wander
    sweeps = rng.randint(1, 3 if dtype == "fp32" else 2)
    if kind in ("batch", "serve"):
        return {"kind": kind, "count": log(4, 96) if kind == "batch" else rng.randint(2, 10),
                "nnz": log(20_000, 2_000_000), "dtype": dtype, "sweeps": sweeps}
    n = rng.choice([3, 3, 4, 5]) if kind != "als" else rng.choice([3, 3, 4])
    nnz = log(2_000, 20_000_000)
    dims = [log(40, 400_000) for _ in range(n)]
    if n > 3:
        dims[-1] = log(2, 400)  # longer tensors have a short, time-like mode
    alpha = rng.choice(["", "1.0", "1.1", "1.2"])
    alphas = [alpha] * n
    if n > 3:
        alphas[-1] = ""
    cells = 1
    for d in dims:
        cells *= d
    nnz = max(1000, min(nnz, cells // 8))
    return {"kind": kind, "dims": "x".join(map(str, dims)), "alphas": ",".join(alphas), "nnz": nnz,
            "rank": rng.choice([8, 10, 16, 16, 24, 32, 32, 48, 64]), "dtype": dtype,
            "values": rng.choice(["uniform", "lognormal"]),
            "sweeps": sweeps if kind == "als" else 0}


# ---- inputs ------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _tensor(g, dims, alphas, nnz, values):
    """(idx, vals): nnz distinct cells in random order (fewer where a skewed
    shape does not yield them in a few rounds)."""
    cdfs = []
    for n, a in zip(dims, alphas):
        # summed on the host: a parallel sum on the device has no fixed order
        w = np.cumsum(np.arange(1, n + 1, dtype=np.float64) ** -a) if a else None
        cdfs.append(torch.from_numpy(w).cuda() if a else None)
    lin = torch.empty(0, dtype=torch.int64, device="cuda")
    count = int(nnz * (2.4 if any(alphas) else 1.2)) + 1024
    for _ in range(6):
        new = torch.zeros(count, dtype=torch.int64, device="cuda")
        for n, c in zip(dims, cdfs):
            if c is None:
                x = torch.randint(0, n, (count,), generator=g, device="cuda")
            else:
                u = torch.rand(count, generator=g, device="cuda", dtype=torch.float64) * c[-1]
                x = torch.searchsorted(c, u, right=True).clamp_max_(n - 1)
            new.mul_(n).add_(x)
        lin = torch.unique(torch.cat([lin, new]))
        if lin.numel() >= nnz:
            break
        count = int((nnz - lin.numel()) * 4) + 4096
    lin = lin[torch.randperm(lin.numel(), generator=g, device="cuda")[:nnz]]
    idx = []
    for n in reversed(dims):
        idx.append((lin % n).to(torch.int32))
        lin = lin // n
    m = idx[0].numel()
    if values == "lognormal":
        vals = torch.empty(m, device="cuda").log_normal_(0.0, 1.0, generator=g)
    else:
        vals = torch.rand(m, generator=g, device="cuda")
    return idx[::-1], vals


def _factors(g, dims, rank):
    return [torch.randn(n, rank, generator=g, device="cuda") for n in dims]


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _flags(case):
    return spm.SPM_FACTOR_BF16 if case["dtype"] == "bf16" else spm.SPM_FACTOR_FP32


def _members(case):
    """Shapes of the tensors of a batch or a job queue: a spread that belongs
    to the case, not to the seed.  Batches: 3 modes of 100 to 20,000 rows,
    ranks 16 and 32.  Queues: 3 or 4 skewed modes of 1,000 to 100,000 rows,
    ranks 8 to 64."""
    out = []
    for t in range(case["count"]):
        def spread(k, lo, hi):  # log-spread, low-discrepancy over the members
            u = (t * 0.6180339887498949 + 0.5 + k * 0.7548776662466927) % 1.0
            return int(round(lo * (hi / lo) ** u))
        if case["kind"] == "batch":
            dims, alphas = [spread(k, 100, 20_000) for k in range(3)], [0.0] * 3
            nnz, rank = spread(3, 1000, case["nnz"]), (16, 32)[t % 2]
        else:
            n = 3 + t % 2
            dims, alphas = [spread(k, 1000, 100_000) for k in range(n)], [1.1] * n
            nnz, rank = spread(4, 10_000, case["nnz"]), (8, 16, 32, 64)[(t // 2) % 4]
        cells = 1
        for d in dims:
            cells *= d
        out.append((dims, alphas, min(nnz, cells // 4), rank))
    return out


def _inputs(case, seed):
    """The tensors of the case with their starting factors, from the seed alone."""
    g = _gen(seed)
    if case["kind"] in ("batch", "serve"):
        out = []
        for dims, alphas, nnz, rank in _members(case):
            idx, vals = _tensor(g, dims, alphas, nnz, "uniform")
            out.append((dims, idx, vals, rank, _factors(g, dims, rank)))
        return out
    dims = [int(d) for d in case["dims"].split("x")]
    alphas = [float(a) if a else 0.0 for a in case["alphas"].split(",")] if case["alphas"] else []
    alphas += [0.0] * (len(dims) - len(alphas))
    idx, vals = _tensor(g, dims, alphas, case["nnz"], case["values"])
    return [(dims, idx, vals, case["rank"], _factors(g, dims, case["rank"]))]


def prepare(case, seed):
    inputs, dt = _inputs(case, seed), _dtype(case)
    s = {"case": case}
    if case["kind"] == "plan":
        s["dims"], s["idx"], s["vals"], s["rank"], _ = inputs[0]
        return s
    if case["kind"] == "serve":
        s["jobs"] = inputs
        return s
    if case["kind"] == "batch":
        s["plans"] = [spm.spmttkrp_plan(d, i, v, r, _flags(case) | spm.SPM_KAPPA(
            max(1, -(-v.numel() // NNZ_PER_PARTITION)))) for d, i, v, r, _ in inputs]
        # every factor a view of one buffer, so that a restart is one copy
        s["init"] = torch.cat([f.reshape(-1) for x in inputs for f in x[4]]).to(dt)
        s["model"] = torch.empty_like(s["init"])
        s["factors"], at = [], 0
        for x in inputs:
            s["factors"].append([])
            for f in x[4]:
                s["factors"][-1].append(s["model"][at:at + f.numel()].view(f.shape))
                at += f.numel()
        s["lam"] = torch.zeros(sum(x[3] for x in inputs), dtype=torch.float64, device="cuda")
        s["fit"] = torch.zeros(len(inputs), dtype=torch.float64, device="cuda")
        return s
    dims, idx, vals, rank, fac = inputs[0]
    s["plan"] = spm.spmttkrp_plan(dims, idx, vals, rank, _flags(case))
    s["factors"] = [f.to(dt) for f in fac]
    if case["kind"] == "mttkrp":
        s["out"] = [torch.empty(n, rank, device="cuda") for n in dims]
    else:
        s["init"] = [f.clone() for f in s["factors"]]
        s["lam"] = torch.zeros(rank, dtype=torch.float64, device="cuda")
        s["fit"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    return s


# ---- one pass ----------------------------------------------------------------

def run(s):
    case = s["case"]
    if case["kind"] == "mttkrp":
        for d, out in enumerate(s["out"]):
            spm.spmttkrp_run(s["plan"], d, s["factors"], out)
        return s["out"]
    if case["kind"] == "als":
        for f, f0 in zip(s["factors"], s["init"]):
            f.copy_(f0)
        spm.cpd_als_reset(s["plan"])
        for _ in range(case["sweeps"]):
            spm.cpd_als_step(s["plan"], s["factors"], s["lam"], s["fit"])
        return {"factors": s["factors"], "weights": s["lam"].to(_dtype(case)), "fit": s["fit"].float()}
    if case["kind"] == "batch":
        s["model"].copy_(s["init"])
        b = spm.spm_batch_create(s["plans"], s["factors"], s["lam"], s["fit"],
                                 max_sweeps=case["sweeps"])
        for _ in range(case["sweeps"]):
            spm.spm_batch_sweep(b)
        out = {"model": s["model"], "weights": s["lam"].to(_dtype(case)), "fit": s["fit"].float()}
        b.destroy()
        return out
    if case["kind"] == "plan":
        p = spm.spmttkrp_plan(s["dims"], s["idx"], s["vals"], s["rank"], _flags(case))
        kappa, units = spm.binding.default_kappa(), spm.SPM_UNITS_PER_PARTITION(s["rank"])
        out = []
        for d in range(len(s["dims"])):
            perm = torch.empty(p.nnz, dtype=torch.int64, device="cuda")
            off = torch.empty(kappa * units + 1, dtype=torch.int64, device="cuda")
            out.append(spm.spmttkrp_plan_permutation(p, d, perm))
            out.append(spm.spmttkrp_plan_work_units(p, d, off))
        p.destroy()
        return out
    server = spm.Server(64 << 30, 64, _flags(case), NNZ_PER_PARTITION)
    ids = [server.submit(d, i, v, r, f, tol=0.0, max_sweeps=case["sweeps"])
           for d, i, v, r, f in s["jobs"]]
    while any(server.step()):
        pass
    out = []
    for j in ids:
        fac, lam = server.result(j)
        out.append(fac + [lam.to(_dtype(case))])
    server.destroy()
    return out


# ---- what a pass cannot do without -------------------------------------------

def work(case):
    if case["kind"] in ("batch", "serve"):
        shapes = [(d, nnz, r) for d, _, nnz, r in _members(case)]
    else:
        shapes = [([int(d) for d in case["dims"].split("x")], case["nnz"], case["rank"])]
    sf = 2 if case["dtype"] == "bf16" else 4
    nbytes = flops = 0
    for dims, nnz, rank in shapes:
        n, rows = len(dims), sum(dims)
        record = 4 * n + 4
        if case["kind"] in ("plan", "serve"):  # read the tensor, write n copies of it and their orders
            nbytes += nnz * record + n * nnz * (record + 4)
        if case["kind"] == "plan":  # the orders as the caller reads them
            nbytes += n * nnz * 8
            continue
        # every mode reads its copy and the other factors and writes one row per index
        passes = max(1, case["sweeps"])
        nbytes += passes * (n * nnz * record + (n - 1) * rows * rank * sf +
                            rows * rank * (4 if case["kind"] == "mttkrp" else sf))
        flops += passes * n * nnz * rank * n
        if case["kind"] != "mttkrp":  # row solves and Grams
            flops += passes * rows * rank * rank * 4
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits -----------------------------------------------------

def _mttkrp64(dims, idx, vals, fac, d):
    out = torch.zeros(dims[d], fac[0].shape[1], dtype=torch.float64, device="cuda")
    step = 1 << 22
    for k in range(0, vals.numel(), step):
        x = vals[k:k + step].double()[:, None]
        for w, f in enumerate(fac):
            if w != d:
                x = x * f[idx[w][k:k + step].long()]
        out.index_add_(0, idx[d][k:k + step].long(), x)
    return out


def _als64(dims, idx, vals, rank, fac, sweeps, dt):
    """CP-ALS with every factor stored in the storage type after its update."""
    fac = [f.to(dt).double() for f in fac]
    grams = [f.T @ f for f in fac]
    lam = fit = None
    for _ in range(sweeps):
        for d in range(len(dims)):
            m = _mttkrp64(dims, idx, vals, fac, d)
            v = torch.ones(rank, rank, dtype=torch.float64, device="cuda")
            for w, g in enumerate(grams):
                if w != d:
                    v = v * g
            z = torch.cholesky_solve(m.T, torch.linalg.cholesky(v)).T
            lam = z.norm(dim=0)
            fac[d] = (z / torch.where(lam > 0, lam, torch.ones_like(lam))).to(dt).double()
            grams[d] = fac[d].T @ fac[d]
        v = torch.ones(rank, rank, dtype=torch.float64, device="cuda")
        for g in grams:
            v = v * g
        norm2 = vals.double().square().sum()
        res = norm2 + lam @ v @ lam - 2 * (lam * (m * fac[-1]).sum(0)).sum()
        fit = 1 - (res.clamp_min(0) / norm2).sqrt()
    return fac, lam, fit.reshape(1)


def exact(case, seed):
    if case["kind"] == "plan":
        return None  # orders and offsets: whole numbers
    inputs, dt = _inputs(case, seed), _dtype(case)
    if case["kind"] == "mttkrp":
        dims, idx, vals, _, fac = inputs[0]
        fac = [f.to(dt).double() for f in fac]
        return [_mttkrp64(dims, idx, vals, fac, d) for d in range(len(dims))]
    got = [_als64(dims, idx, vals, rank, fac, case["sweeps"], dt)
           for dims, idx, vals, rank, fac in inputs]
    if case["kind"] == "als":
        return {"factors": got[0][0], "weights": got[0][1], "fit": got[0][2]}
    if case["kind"] == "batch":
        return {"model": torch.cat([f.reshape(-1) for x in got for f in x[0]]),
                "weights": torch.cat([x[1] for x in got]), "fit": torch.cat([x[2] for x in got])}
    return [list(x[0]) + [x[1]] for x in got]
