"""What users of this library have it do, as cases that can be timed and compared.

A case calls one public entry point of the Python binding on data of a stated size:
  fit         lingam.fit, one dataset -> causal order and B;
  bootstrap   lingam.fit_bootstrap, resamples of one dataset -> their orders and Bs;
  batch       lingam.fit_batch, datasets of uneven sizes -> their orders and Bs;
  covariance  lingam.covariance, the covariance of the normalised rows alone.

The data are LiNGAM samples X = B X + N (B strictly lower triangular in a random causal
order) with the library's own noise families (uniform, Laplace, signed powers of a Gaussian).
Every variable has its predecessor in the causal order among its parents and each earlier
variable with a small probability besides, so that the causal order is unique: two correct
implementations then find the same order, where a graph with several exogenous variables
leaves near-ties that the rounding of a sum decides.  Rows have unit variance, as users
usually bring them.
"""
import math

import numpy as np
import torch

from paper_2109_13993_gb300 import lingam

K1, K2, BETA = 79.047, 7.4129, 0.37457   # the constants of the entropy approximation, as printed in the paper


def listed():
    return [
        # the smallest fit of the benchmark configurations: launches and latency
        dict(name="fit p20 n2000", kind="fit", p=20, n=2000, precision="mixed", dtype="float32", host=False),
        # plain DirectLiNGAM in FP64, the first benchmark configuration
        dict(name="fit fp64 p20 n2000", kind="fit", p=20, n=2000, precision="fp64", dtype="float64", host=False),
        # odd sizes in FP64
        dict(name="fit fp64 p65 n2001", kind="fit", p=65, n=2001, precision="fp64", dtype="float64", host=False),
        # an ordinary single dataset, the second configuration
        dict(name="fit p100 n10000", kind="fit", p=100, n=10000, precision="mixed", dtype="float32", host=False),
        # a user's numpy array of doubles, odd sizes, copied to the device inside the call
        dict(name="fit host p257 n3001", kind="fit", p=257, n=3001, precision="mixed", dtype="float64", host=True),
        # the third configuration
        dict(name="fit p300 n5000", kind="fit", p=300, n=5000, precision="mixed", dtype="float32", host=False),
        # few variables, long recordings
        dict(name="fit p50 n100000", kind="fit", p=50, n=100000, precision="mixed", dtype="float32", host=False),
        # the large single dataset of the headline benchmark
        dict(name="fit p1000 n10000", kind="fit", p=1000, n=10000, precision="mixed", dtype="float32", host=False),
        # the fourth configuration: bootstrap confidence of one dataset, and many uneven datasets
        dict(name="bootstrap 256 p50 n2000", kind="bootstrap", p=50, n=2000, count=256),
        dict(name="batch 64 uneven", kind="batch", count=64, p_lo=20, p_hi=120, n_lo=500, n_hi=8000),
        # the covariance alone, on the tensor cores and in FP64
        dict(name="covariance p1000 n10000", kind="covariance", p=1000, n=10000, precision="mixed", dtype="float32"),
        dict(name="covariance fp64 p300 n5000", kind="covariance", p=300, n=5000, precision="fp64", dtype="float64"),
    ]


def work(case):
    """Every fit compares its roots with every variable left (each pair of variables once: both
    scores of a pair come from one evaluation), which also is the least that shows the others not
    to be roots.  A pair and sample: two residuals (2 operations each), for each its two moments
    (about 16, an exponential or a logarithm counted as one)."""
    if case["kind"] == "covariance":
        p, n = case["p"], case["n"]
        return {"bytes": p * n * (4 if case["dtype"] == "float32" else 8) + 8 * p * p, "flops": float(p) * p * n}
    if case["kind"] == "batch":
        each = list(zip(*_sizes(case)))
    else:
        each = [(case["p"], case["n"])] * case.get("count", 1)
    pairs = sum(p * (p - 1) / 2.0 * n for p, n in each)
    read = sum(p * n for p, n in each) * (8 if case.get("dtype") == "float64" else 4)
    if case["kind"] == "bootstrap":   # one dataset, and the resamples' indices
        read = case["p"] * case["n"] * 4 + case["count"] * case["n"] * 4
    return {"bytes": read + sum(4 * p + 8 * p * p for p, _ in each), "flops": 36.0 * pairs}


def tolerance(case):
    """Orders are the same; B and the covariance carry the rounding of the rows: to FP32 on the
    mixed path (2e-8 to 4e-8 measured against 64 bits), FP64 sums otherwise (5e-15)."""
    if case.get("precision") == "fp64":
        return {"rel": 1e-13, "differ": 0.0}
    return {"rel": 4e-7, "differ": 0.0}


def _log_int(rng, lo, hi):
    """A whole number between lo and hi, evenly over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "fit64", "bootstrap", "batch", "covariance", "covariance"])
    if kind == "fit":
        p = _log_int(rng, 12, 900)
        n = _log_int(rng, max(2000, 8 * p), min(100000, 9000000 // p))   # fewer samples leave near-ties
        return dict(kind="fit", p=p, n=n, precision="mixed", dtype=rng.choice(["float32", "float32", "float64"]),
                    host=rng.random() < 0.25)
    if kind == "fit64":
        p = _log_int(rng, 8, 80)
        return dict(kind="fit", p=p, n=_log_int(rng, 1500, 6000), precision="fp64", dtype="float64",
                    host=rng.random() < 0.25)
    if kind == "bootstrap":
        p = _log_int(rng, 12, 120)
        return dict(kind="bootstrap", p=p, n=_log_int(rng, 1000, 5000), count=_log_int(rng, 32, 400))
    if kind == "batch":
        p_lo, n_lo = _log_int(rng, 10, 60), _log_int(rng, 500, 4000)
        return dict(kind="batch", count=_log_int(rng, 8, 100), p_lo=p_lo, p_hi=p_lo + _log_int(rng, 10, 100),
                    n_lo=n_lo, n_hi=n_lo + _log_int(rng, 500, 8000))
    precision = rng.choice(["mixed", "mixed", "fp64"])
    p = _log_int(rng, 20, 1000 if precision == "mixed" else 400)
    n = _log_int(rng, 1000, min(100000, (9000000 if precision == "mixed" else 2000000) // p))
    return dict(kind="covariance", p=p, n=n, precision=precision,
                dtype=rng.choice(["float32", "float64"]) if precision == "mixed" else "float64")


# ------------------------------------------------------------------ inputs
def _dataset(p, n, g):
    """p x n LiNGAM samples (float64, on the GPU), rows of unit variance; see the module's docstring."""
    dev = g.device
    rand = lambda *s: torch.rand(*s, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
    normal = torch.randn(p, n, generator=g, device=dev, dtype=torch.float64)
    unif = rand(p, n)
    lap = unif - 0.5
    lap = -torch.sign(lap) * torch.log1p(-2 * lap.abs()) / math.sqrt(2.0)
    power = torch.sign(normal) * normal.abs() ** (1.4 + 0.6 * rand(p, 1))
    kind = torch.randint(0, 3, (p, 1), generator=g, device=dev)
    e = torch.where(kind == 0, (2 * unif - 1) * math.sqrt(3.0), torch.where(kind == 1, lap, power))
    e = e / e.std(dim=1, keepdim=True)
    # weights in causal positions: the predecessor, and one more parent on average
    sign = lambda *s: torch.sign(rand(*s) - 0.5)  # noqa: E731
    extra = torch.where(rand(p, p) < 2.0 / max(p - 1, 1), (0.15 + 0.25 * rand(p, p)) * sign(p, p), 0.0)
    w = torch.tril(extra, -2)
    if p > 1:
        at = torch.arange(1, p, device=dev)
        w[at, at - 1] = (0.6 + 0.25 * rand(p - 1)) * sign(p - 1)
    total = w.abs().sum(dim=1, keepdim=True)
    w = torch.where(total > 0.95, w * (0.95 / total.clamp_min(1e-30)), w)   # bounded variance along the order
    eye = torch.eye(p, device=dev, dtype=torch.float64)
    x = torch.linalg.solve_triangular(eye - w, e, upper=False, unitriangular=True)
    x = x / x.std(dim=1, keepdim=True)
    return x[torch.randperm(p, generator=g, device=dev)].contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _sizes(case):
    """The batch's sizes: uniform in the case's ranges, the same for every seed."""
    rng = np.random.default_rng([case[k] for k in ("count", "p_lo", "p_hi", "n_lo", "n_hi")])
    ps = rng.integers(case["p_lo"], case["p_hi"] + 1, case["count"])
    ns = rng.integers(case["n_lo"], case["n_hi"] + 1, case["count"])
    return [int(p) for p in ps], [int(n) for n in ns]


def _inputs(case, seed):
    g = _generator(seed)
    if case["kind"] == "batch":
        return [_dataset(p, n, g).float() for p, n in zip(*_sizes(case))]
    x = _dataset(case["p"], case["n"], g)
    if case["kind"] == "bootstrap":
        idx = torch.randint(0, case["n"], (case["count"], case["n"]), generator=g, device="cuda", dtype=torch.int32)
        return x.float(), idx
    x = x.to(getattr(torch, case["dtype"]))
    return x.cpu().numpy() if case.get("host") else x


def prepare(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    if kind == "batch":
        ws = lingam.batch_workspace([d.shape[0] for d in x], [d.shape[1] for d in x])
    elif kind == "bootstrap":
        x, idx = x
        o, _ = lingam.make_opts("mixed", np.float32)
        ws = lingam.alloc_workspace(lingam.load().lingam_workspace_size_bootstrap(case["p"], case["n"], case["count"], o))
        return dict(kind=kind, x=x, idx=idx, ws=ws)
    else:
        ws = lingam.alloc_workspace(lingam.workspace_size(case["p"], case["n"], case["precision"], np.dtype(case["dtype"])))
    return dict(kind=kind, x=x, ws=ws, precision=case.get("precision"))


def run(state):
    kind = state["kind"]
    if kind == "fit":
        r = lingam.fit(state["x"], precision=state["precision"], workspace=state["ws"])
        return {"order": r.order, "B": r.B}
    if kind == "covariance":
        return lingam.covariance(state["x"], precision=state["precision"], workspace=state["ws"])[0]
    if kind == "bootstrap":
        r = lingam.fit_bootstrap(state["x"], state["idx"], workspace=state["ws"])
    else:
        r = lingam.fit_batch(state["x"], workspace=state["ws"])
    return {"status": r.statuses, "order": np.concatenate(r.orders), "B": np.concatenate([b.ravel() for b in r.Bs])}


# ------------------------------------------------------------------ the same in 64 bits
def _log_cosh_mean(u):
    a = u.abs()
    return (a + torch.log1p(torch.exp(-2 * a)) - math.log(2.0)).mean(dim=-1)


def _entropy(u):
    """Eq. HApp without the constant H(nu), over the last axis."""
    return -K1 * (_log_cosh_mean(u) - BETA) ** 2 - K2 * (u * torch.exp(-0.5 * u * u)).mean(dim=-1) ** 2


def _normalised(x):
    x = x - x.mean(dim=1, keepdim=True)
    return x / x.std(dim=1, keepdim=True)


def _exact_fit(x):
    """DirectLiNGAM of x (p x n, float64), every pair compared: the order (a list) and B."""
    p, n = x.shape
    left = torch.arange(p, device=x.device)
    z, order = _normalised(x), []
    while len(left) > 1:
        r = len(left)
        h, rho = _entropy(z), z @ z.T / (n - 1)
        ii, jj = torch.triu_indices(r, r, 1, device=x.device)
        measure = []
        for c in range(0, len(ii), max(1, 20_000_000 // n)):
            i, j = ii[c:c + max(1, 20_000_000 // n)], jj[c:c + max(1, 20_000_000 // n)]
            q = rho[i, j][:, None]
            s = torch.sqrt(1 - q * q)
            a, b = _entropy((z[i] - q * z[j]) / s), _entropy((z[j] - q * z[i]) / s)
            measure.append((h[j] + a) - (h[i] + b))
        measure = torch.cat(measure)
        score = torch.zeros(r, dtype=x.dtype, device=x.device)
        score.index_add_(0, ii, measure.clamp(max=0) ** 2)
        score.index_add_(0, jj, measure.clamp(min=0) ** 2)
        k = int(score.argmin())
        order.append(int(left[k]))
        keep = torch.arange(r, device=x.device) != k
        z = _normalised(z[keep] - rho[keep, k][:, None] * z[k])
        left = left[keep]
    order.append(int(left[0]))
    return order, _exact_b(x, order)


def _exact_b(x, order):
    """Least squares of every variable on its predecessors in the order."""
    xc = x - x.mean(dim=1, keepdim=True)
    at = torch.tensor(order, device=x.device)
    low = torch.linalg.cholesky((xc @ xc.T / (x.shape[1] - 1))[at][:, at])
    eye = torch.eye(len(order), dtype=x.dtype, device=x.device)
    bk = eye - torch.diagonal(low)[:, None] * torch.linalg.solve_triangular(low, eye, upper=False)
    b = torch.zeros_like(bk)
    b[at[:, None], at[None, :]] = torch.tril(bk, -1)
    return b


def _pair_samples(p, n):
    """Pairs compared over all iterations of an unpruned fit, times the samples."""
    return (p * p * p - p) / 6.0 * n


EXACT_MOST = 1.0e10   # pair-samples that the 64-bit path takes a few seconds for


def exact(case, seed):
    x = _inputs(case, seed)
    if case["kind"] == "covariance":
        z = _normalised(x.double())
        return (z @ z.T / (case["n"] - 1)).cpu().numpy()
    if case["kind"] == "fit":
        if _pair_samples(case["p"], case["n"]) > EXACT_MOST:
            return None
        order, b = _exact_fit(torch.as_tensor(x, device="cuda").double())
        return {"order": np.array(order, dtype=np.int32), "B": b.cpu().numpy()}
    if case["kind"] == "bootstrap":
        if case["count"] * _pair_samples(case["p"], case["n"]) > EXACT_MOST:
            return None
        many = [x[0].double()[:, i.long()] for i in x[1]]
    else:
        if sum(_pair_samples(p, n) for p, n in zip(*_sizes(case))) > EXACT_MOST:
            return None
        many = [d.double() for d in x]
    fits = [_exact_fit(d) for d in many]
    return {"status": None, "order": np.concatenate([np.array(o, dtype=np.int32) for o, _ in fits]),
            "B": torch.cat([b.reshape(-1) for _, b in fits]).cpu().numpy()}
