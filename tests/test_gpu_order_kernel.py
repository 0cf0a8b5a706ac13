"""The ordering kernel, its factor-based B fit and the covariance kernels at the sizes where their splits
change: units and the last, partial one (128 / 64 samples a step), rows of a worker (32), columns
(4 ... 16), the controller's warps, in-place and permuted factors (128 variables), the lines between
ordering and tile kernels (unpruned 80 variables or 24 samples a variable; the largest sizes; fits
that are handed over), queued problems of a batch (more than 304), tiles and parts of the
covariance (128, 8; 32 on the FP64 path)."""
import functools

import numpy as np
import pytest

import oracle
from paper_2109_13993_gb300 import lingam, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2109_13993_gb300 import build
    build.build()
    lingam.load()
    oracle.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _data(p, n, seed):
    return synth.lingam_dataset(p, n, min(1.0, 3.0 / max(p - 1, 1)), seed).X


def _dev(X, dtype):
    return torch.tensor(np.ascontiguousarray(X), dtype=dtype, device="cuda")


SIZES = [(1, 9), (2, 5), (3, 40), (4, 63), (5, 64), (9, 65), (16, 127), (17, 128), (18, 129), (33, 257), (34, 1023),
         (40, 1025), (65, 300)]


@pytest.mark.parametrize("p,n", SIZES)
@pytest.mark.parametrize("prune", [True, False])
def test_fp64_fit_matches_oracle(p, n, prune):
    # FP64 throughout: 1e-10 relative on scores and B, as for the whole FP64 path
    X = _data(p, n, 100 * p + n)
    o_order, o_B, o_S = oracle.fit(X)
    f = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=prune)
    assert np.array_equal(f.order, o_order)
    want = np.array([o_S[k, o_order[k]] for k in range(p)])
    assert np.all(np.abs(f.root_score - want) <= 1e-10 * np.abs(want) + 1e-14)
    assert np.abs(f.B - o_B).max() <= 1e-10 * max(1.0, np.abs(o_B).max())


@pytest.mark.parametrize("p,n", SIZES + [(80, 500), (81, 500), (100, 2399), (100, 2400), (127, 500), (128, 500), (129, 500),
                                         (160, 640), (161, 640)])
def test_mixed_scores_and_pruned_roots(p, n):
    # every score within the mixed path's 1e-4 of the oracle; the killer pairs change no root's score.
    # Equal up to the FP32 rounding of I, 1e-6 absolute: S = sum of m squares I_j^2 moves by at most
    # 2e-6 sum |I_j| + m 1e-12 <= 2e-6 sqrt(m S) + m 1e-12 (Cauchy-Schwarz)
    X = _data(p, n, 100 * p + n).astype(np.float32)
    o_order, o_B, o_S = oracle.fit(X.astype(np.float64))
    full = lingam.fit(_dev(X, torch.float32), prune=False, forced_order=o_order, want_scores=True)
    m = ~np.isnan(o_S)
    assert np.array_equal(m, ~np.isnan(full.scores))
    assert np.abs(full.scores[m] - o_S[m]).max() <= 1e-4
    assert np.abs(full.B - o_B).max() <= 1e-4 * max(1.0, np.abs(o_B).max())
    pruned = lingam.fit(_dev(X, torch.float32), forced_order=o_order)
    left = p - 1 - np.arange(p)
    assert np.all(np.abs(pruned.root_score - full.root_score) <= 2e-6 * np.sqrt(left * full.root_score) + left * 1e-12)
    assert np.abs(pruned.B - full.B).max() <= 1e-12 * max(1.0, np.abs(o_B).max())


def _b_long_double(X, order):
    """B of X in a given causal order, by elimination in long double."""
    L = np.longdouble
    x = X[order].astype(L)
    x = x - x.mean(axis=1, keepdims=True)
    S, p = x @ x.T, len(order)
    low, d = np.eye(p, dtype=L), np.zeros(p, dtype=L)
    for k in range(p):
        d[k] = S[k, k]
        low[k + 1:, k] = S[k + 1:, k] / d[k]
        S[k + 1:, k + 1:] -= np.outer(low[k + 1:, k], low[k + 1:, k]) * d[k]
    inv = np.eye(p, dtype=L)
    for i in range(1, p):
        inv[i, :i] = -low[i, :i] @ inv[:i, :i]
    B = np.zeros((p, p), dtype=L)
    B[np.ix_(order, order)] = np.eye(p, dtype=L) - inv
    return B


def test_fp64_b_is_no_further_off_than_the_cholesky():
    # B from the ordering's elimination against the tile kernels' Cholesky, both from the same covariance:
    # mean logarithm of their errors over 24 graphs
    err = []
    for seed in range(24):
        X = _data(50, 500, seed)
        a = lingam.fit(_dev(X, torch.float64), precision="fp64")
        b = lingam.fit(_dev(X, torch.float64), precision="fp64", tile_i=32, tile_j=32, forced_order=a.order)
        ref = _b_long_double(X, a.order)
        err.append([np.linalg.norm((r.B - ref).astype(np.float64)) for r in (a, b)])
    here, cholesky = np.exp(np.log(err).mean(axis=0))
    assert here <= cholesky, (here, cholesky)


def _near_tie(seed, weight):
    """Six variables whose second iteration ends in a near tie: weight moves the scores, in steps far
    below their gap."""
    p, n = 6, 300
    X = np.stack([synth.noise(synth.Stream(seed, v), (synth.NOISE_LAPLACE, synth.NOISE_UNIFORM)[v % 2], n)
                  for v in range(p)])
    W = np.tril(2 * synth.Stream(seed, 9).uniform(p * p).reshape(p, p) - 1, -1)
    W[5, 4] = weight
    for i in range(p):
        X[i] += W[i, :i] @ X[:i]
    return X


@pytest.mark.parametrize("seed,weight", [(187, 0.299236631094986), (327, -0.5675924855453444),
                                         (358, -0.4380522633860032), (1345, 0.04396862919510971),
                                         (1399, -0.6748515948032312)])
def test_fp64_pruning_is_exact_at_a_near_tie(seed, weight):
    # the lowest score lies 3e-8 below the next and comes from a single pair, whose square rounded to the
    # nearest FP32 value is above the next score: as a killer's share it has to be rounded down (seed 327
    # is one where it is the killer's)
    X = _near_tie(seed, weight)
    o_order, _, o_S = oracle.fit(X)
    low, second = np.sort(o_S[1][~np.isnan(o_S[1])])[:2]
    assert 1e-8 < (second - low) / low < 1e-7
    full = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=False)
    pruned = lingam.fit(_dev(X, torch.float64), precision="fp64")
    assert np.array_equal(full.order, o_order)
    assert np.array_equal(pruned.order, o_order)
    assert 0.0 <= pruned.margin_lb[1] <= (second - low) * (1 + 1e-3)   # (scores to 1e-10: 3e-3 of the gap at most)


@pytest.mark.parametrize("p,precision,gram,factor", [(20, "mixed", 3, 1), (128, "mixed", 3, 1), (129, "mixed", 3, 2),
                                                     (20, "fp64", 2, 1), (129, "fp64", 2, 2), (800, "fp64", 1, 0)])
def test_kernel_launches_reported(p, precision, gram, factor):
    # the rows, the covariance (FP64: without splits of the samples from 25 x 25 tiles of 32 on, one kernel),
    # the ordering, B (above 128 variables from a permuted copy)
    X = _dev(_data(min(p, 200), 900, 60 + p), torch.float64)
    if factor:
        r = lingam.fit(X[:p], precision=precision)
        assert r.kernel_launches == 1 + gram + 1 + factor
        assert lingam.fit(X[:p], precision=precision, want_B=False).kernel_launches == 1 + gram + 1
    else:
        X = torch.randn(p, 900, dtype=torch.float64, device="cuda")
    assert lingam.covariance(X[:p], precision=precision)[1]["kernel_launches"] == 1 + gram


@pytest.mark.parametrize("p,max_iters", [(1, 0), (2, 0), (20, 0), (20, 7)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_iteration_times_do_not_hold_what_the_workspace_held(p, max_iters, precision):
    X = _dev(_data(p, 700, 50 + p), torch.float64)
    ws = lingam.alloc_workspace(lingam.workspace_size(p, 700, precision, np.float64))
    ws.fill_(0xff)   # NaN as doubles
    r = lingam.fit(X, precision=precision, timing=True, max_iters=max_iters, workspace=ws)
    t = r.t_pair_iter_ms
    assert np.all(np.isfinite(t)) and np.all(t >= 0.0)
    assert t.sum() <= r.times_ms["pair"]
    assert np.all(t[:(max_iters or p - 1)] > 0.0)


@pytest.mark.parametrize("p,n", [(50, 2000), (150, 2000), (161, 700)])
@pytest.mark.parametrize("start", ["low", "high"])
def test_threshold_schedule_compares_no_more_pairs_than_the_tile_kernels(p, n, start):
    # the killer pairs bound the scores under the paper's threshold schedule too; the roots are the same
    X = _dev(_data(p, n, 1), torch.float32)
    ref = lingam.fit(X)
    rs = ref.root_score[ref.root_score > 0]
    gamma0 = float(1e-3 * rs.min() if start == "low" else 10.0 * rs.max())
    here = lingam.fit(X, gamma0=gamma0, forced_order=ref.order)
    tiles = lingam.fit(X, gamma0=gamma0, forced_order=ref.order, tile_i=64, tile_j=32)
    assert here.pairs_total < tiles.pairs_total
    assert (here.threshold_updates > 0) == (tiles.threshold_updates > 0) == (start == "low")
    assert np.allclose(here.root_score, ref.root_score, rtol=1e-6, atol=1e-9)
    free = lingam.fit(X, gamma0=gamma0)
    assert np.array_equal(free.order, ref.order)


@pytest.mark.parametrize("sizes", [[(64, 600)] * 2, [(65, 600)] * 2, [(40, 1025)] * 3, [(70, 512)] * 3, [(70, 512)] * 4,
                                   [(70, 513)] * 4, [(20, 8000)] * 2, [(70, 8000)], [(70, 7999)], [(128, 700), (3, 40)],
                                   [(129, 513), (9, 100)], [(129, 512), (9, 100)], [(161, 600), (9, 100)], [(1, 9), (2, 5)]])
@pytest.mark.parametrize("tile", [0, 1])
def test_unpruned_batches_on_either_side_of_the_routes(sizes, tile):
    # ordering kernel, pairs by warps and tiles: scores of every variable against FP64, B against the single
    # fit's.  1e-4 is the mixed path's stated tolerance
    Xs = [_data(p, n, 9000 + 10 * k + p).astype(np.float32) for k, (p, n) in enumerate(sizes)]
    got = lingam.fit_batch([_dev(X, torch.float32) for X in Xs], prune=False, want_scores=True, tile_i=tile, tile_j=tile)
    assert got.status == lingam.LINGAM_OK
    for X, order, B, S in zip(Xs, got.orders, got.Bs, got.scores):
        ref = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=False, forced_order=order, want_scores=True)
        m = ~np.isnan(ref.scores)
        assert np.array_equal(m, ~np.isnan(S))
        assert np.abs(S[m] - ref.scores[m]).max() <= 1e-4
        assert np.abs(B - ref.B).max() <= 1e-4 * max(1.0, np.abs(ref.B).max())


def _common_causes(p, n, causes, seed):
    """Independent variables but for `causes` of them, each a parent of all the others."""
    e = np.random.default_rng(seed).laplace(size=(p, n))
    for c in range(causes):
        e[c + 1:] += 0.8 * e[c]
    return e.astype(np.float32)


@functools.lru_cache(maxsize=None)
def _common_causes_fp64(p, n, causes, seed):
    X = _common_causes(p, n, causes, seed)
    return X, lingam.fit(_dev(X, torch.float64), precision="fp64", prune=False, want_scores=True)


def _handed_over_at(res, p, want_B=True):
    """Iteration from which tile kernels ran: rows, covariance (3), ordering, the step between, an iteration
    each, B's two kernels tried before and four after."""
    return p - (res.kernel_launches - 6 - (6 if want_B else 0))


@pytest.mark.parametrize("kw", [{}, {"gamma0": 1.0}, {"prior": True}, {"timing": True}, {"split_n": 2}])
def test_hand_over_to_the_tile_kernels(kw):
    # many independent variables: no killer pairs to speak of.  Scores along FP64's order within the mixed
    # path's 1e-4 before and behind the iteration, at even and odd ones (the rows lie in either copy)
    p, n, at = 400, 640, set()
    for causes in (0, 1, 2, 5):
        X, full = _common_causes_fp64(p, n, causes, 70 + causes)
        opts = dict(kw)
        if opts.pop("prior", None):
            opts["prior"] = np.zeros((p, p), dtype=np.int8)
            opts["prior"][full.order[200], full.order[0]] = opts["prior"][full.order[-1], full.order[100]] = 1
        got = lingam.fit(_dev(X, torch.float32), forced_order=full.order, want_scores=True, **opts)
        it0 = _handed_over_at(got, p)
        assert 5 <= it0 < 30
        at.add(it0 % 2)
        m = ~np.isnan(got.scores)
        assert np.abs(got.scores[m] - full.scores[m]).max() <= 1e-4
        assert m[:-1].sum(axis=1).min() >= 2
        if "gamma0" not in kw:
            # a variable left out is not the root: its score is above the lowest complete one
            low = np.where(m, got.scores, np.inf).min(axis=1)
            out = ~m & ~np.isnan(full.scores)
            if "prior" not in kw:
                assert np.all(np.where(out, full.scores, np.inf).min(axis=1) >= low - 1e-6)
        assert np.abs(got.root_score - full.root_score).max() <= 1e-6
        assert np.abs(got.B - full.B).max() <= 1e-4 * max(1.0, np.abs(full.B).max())
        assert sorted(lingam.fit(_dev(X, torch.float32), **opts).order.tolist()) == list(range(p))
        if "timing" in kw:
            t = got.t_pair_iter_ms
            assert np.all(np.isfinite(t)) and np.all(t[:-1] > 0.0) and t.sum() <= got.times_ms["order"]
    assert at == ({1} if "gamma0" in kw else {0, 1})   # (nothing is pruned below 1: iteration 5 each time)


def test_hand_over_within_a_bounded_number_of_iterations():
    p, n = 400, 640
    X = _dev(_common_causes(p, n, 1, 71), torch.float32)
    ref = lingam.fit(X)
    it0 = _handed_over_at(ref, p)
    for iters in (it0 - 1, it0, it0 + 1, it0 + 2):
        part = lingam.fit(X, max_iters=iters)
        assert np.array_equal(part.order[:iters], ref.order[:iters]) and np.all(part.order[iters:] == -1)
        assert np.array_equal(part.root_score[:iters], ref.root_score[:iters])
        assert part.kernel_launches == 5 + (iters > it0) * (1 + iters - it0)


# padded samples p x ld (ld a multiple of 128) just below and above the sizes where the units change: 64 and
# 128 samples at 2^16, 128 and 256 at 2^18 (FP64), 256 and 512 at 2^18, 512 and 1024 at 2^22 (mixed); a last
# unit that is not full; samples for several staged passes of a worker (split_n = 1); candidates for the
# several-warp selection (more than 256)
@pytest.mark.parametrize("p,n,split_n", [(40, 1500, 0), (40, 1601, 0), (64, 3967, 0), (64, 4090, 0), (9, 70001, 1)])
def test_fp64_units(p, n, split_n):
    X = _data(p, n, 300 + p)
    o_order, o_B, o_S = oracle.fit(X)
    for prune in (True, False):
        f = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=prune, forced_order=o_order, split_n=split_n)
        want = np.array([o_S[k, o_order[k]] for k in range(p)])
        assert np.all(np.abs(f.root_score - want) <= 1e-10 * np.abs(want) + 1e-14)
        assert np.abs(f.B - o_B).max() <= 1e-10 * max(1.0, np.abs(o_B).max())


@pytest.mark.parametrize("p,n,split_n", [(64, 3967, 0), (64, 4090, 0), (41, 102200, 0), (41, 102300, 0), (9, 200001, 1),
                                         (257, 700, 0), (258, 513, 0), (300, 900, 0)])
def test_mixed_units_and_selection(p, n, split_n):
    X = _data(p, n, 300 + p).astype(np.float32)
    ref = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=False, want_scores=True)
    got = lingam.fit(_dev(X, torch.float32), forced_order=ref.order, want_scores=True, split_n=split_n)
    m = ~np.isnan(got.scores)
    assert not np.any(m & np.isnan(ref.scores))
    assert np.abs(got.scores[m] - ref.scores[m]).max() <= 1e-4
    left = p - 1 - np.arange(p)   # (the bound of test_mixed_scores_and_pruned_roots)
    assert np.all(np.abs(got.root_score - ref.root_score) <= 2e-6 * np.sqrt(left * ref.root_score) + left * 1e-12)
    assert np.abs(got.B - ref.B).max() <= 1e-4 * max(1.0, np.abs(ref.B).max())


def test_mixed_batch_units():
    # a batch's units of 1024 samples with a last one that is not full
    Xs = [_data(p, n, 400 + p).astype(np.float32) for p, n in [(20, 5001), (33, 2047), (9, 1025), (50, 3333), (7, 1023)]]
    got = lingam.fit_batch([_dev(X, torch.float32) for X in Xs], want_scores=True)
    for X, order, S in zip(Xs, got.orders, got.scores):
        ref = lingam.fit(_dev(X, torch.float64), precision="fp64", prune=False, forced_order=order, want_scores=True)
        m = ~np.isnan(S)
        assert m[:-1].sum(axis=1).min() >= 1
        assert np.abs(S[m] - ref.scores[m]).max() <= 1e-4


def _chain(p, n, seed):
    X = np.random.default_rng(seed).laplace(size=(p, n))
    for i in range(1, p):
        X[i] += 0.7 * X[i - 1]
    return X[np.random.default_rng(seed + 1).permutation(p)]


# the last sizes of 16, 12, 8 and 4 columns a wave and the first ones below (controller state and measures
# share 220 KB), and the first sizes for the tile kernels
@pytest.mark.parametrize("p,precision", [(1706, "mixed"), (1707, "mixed"), (1942, "mixed"), (1943, "mixed"), (2252, "mixed"),
                                         (2253, "mixed"), (2681, "mixed"), (2682, "mixed"), (1116, "fp64"), (1117, "fp64"),
                                         (1641, "fp64"), (2146, "fp64")])
def test_largest_single_fits_against_the_tile_kernels(p, precision):
    X = _dev(_chain(p, 192, p), torch.float32 if precision == "mixed" else torch.float64)
    kw = dict(precision=precision, max_iters=4, want_scores=True, want_B=False)
    tiles = lingam.fit(X, tile_i=32, tile_j=32, **kw)
    order = tiles.order[:4].tolist()
    forced = np.array(order + sorted(set(range(p)) - set(order)), dtype=np.int32)
    got = lingam.fit(X, forced_order=forced, **kw)
    assert got.kernel_launches <= tiles.kernel_launches - (0 if p == 2682 else 3)
    m = ~np.isnan(got.scores[:4]) & ~np.isnan(tiles.scores[:4])
    assert m.sum(axis=1).min() >= 1
    s = tiles.scores[:4][m]
    bound = 2e-6 * np.sqrt(p * s) + p * 1e-12 if precision == "mixed" else 1e-10 * s + 1e-14
    assert np.all(np.abs(got.scores[:4][m] - s) <= bound)
    want = tiles.root_score[:4]
    assert np.all(np.abs(got.root_score[:4] - want) <= (2e-6 * np.sqrt(p * want) + p * 1e-12 if precision == "mixed" else 1e-10 * want))


def test_b_of_a_large_fit():
    # the permuted factor, two columns of 2100 doubles a CTA
    p, n = 2100, 8000   # (enough samples that it is not handed over)
    X = _chain(p, n, 5).astype(np.float32)
    got = lingam.fit(_dev(X, torch.float32))
    assert got.kernel_launches == 7
    x = X[got.order].astype(np.float64)
    low = np.linalg.cholesky(np.cov(x))
    want = np.eye(p) - np.diag(low)[:, None] * np.linalg.inv(low)
    B = got.B[np.ix_(got.order, got.order)]
    assert np.all(np.triu(B) == 0.0)
    assert np.abs(B - np.tril(want, -1)).max() <= 1e-4 * np.abs(want).max()


@pytest.mark.parametrize("p", [332, 333, 844, 845, 1100, 1101])
def test_largest_problems_of_a_batch(p):
    # 16, 12, 8 and 4 columns a wave in 108 KB, and the first size for tiles
    X = _dev(_chain(p, p + 200, p), torch.float32)
    small = _dev(_chain(12, 300, 1), torch.float32)
    got = lingam.fit_batch([X, small], want_report=True)
    assert got.status == lingam.LINGAM_OK
    one = lingam.fit(X, forced_order=got.orders[0])
    left = p - 1 - np.arange(p)
    s = one.root_score
    assert np.all(np.abs(got.root_scores[0] - s) <= 4e-6 * np.sqrt(left * s) + left * 4e-12)   # (both rounded)
    assert np.abs(got.Bs[0] - one.B).max() <= 1e-9 * np.abs(one.B).max()
    assert np.array_equal(got.orders[1], lingam.fit(small).order)


def test_batch_with_queued_problems_matches_oracle():
    # more problems than CTA slots, of 2 ... 13 variables, one large enough for a group of its own
    Xs = [_data(2 + k % 12, 40 + 17 * (k % 23), 7000 + k) for k in range(330)] + [_data(60, 3001, 8000)]
    got = lingam.fit_batch([_dev(X, torch.float64) for X in Xs], precision="fp64")
    assert got.status == lingam.LINGAM_OK
    for X, order, B in zip(Xs, got.orders, got.Bs):
        o_order, o_B, _ = oracle.fit(X, want_scores=False)
        assert np.array_equal(order, o_order)
        assert np.abs(B - o_B).max() <= 1e-10 * max(1.0, np.abs(o_B).max())


@pytest.mark.parametrize("p", [1, 7, 8, 9, 31, 32, 33, 127, 128, 129, 136])
@pytest.mark.parametrize("n", [3, 64, 65, 511, 577])
def test_covariance_at_tile_and_part_edges(p, n):
    X = np.random.default_rng(1000 * p + n).standard_normal((p, n))
    X32 = X.astype(np.float32)
    ref = oracle.covariance(X32.astype(np.float64))
    got = lingam.covariance(_dev(X32, torch.float32))[0]
    # rows rounded to FP32 (2^-24 relative), their tails off by 2^-27 of 2^e <= 2 max |x| and the tails'
    # product, 2^-30 of 2^(e_i + e_j), left out; max |x| <= sqrt(n - 1), sums by the Cauchy-Schwarz inequality
    tol = 2 * (2.0**-24 + 2.0**-26 * np.sqrt(n - 1)) + 2.0**-28 * (n - 1)
    assert np.abs(got - ref).max() <= tol
    ref = oracle.covariance(X)
    got = lingam.covariance(_dev(X, torch.float64), precision="fp64")[0]
    # the rows' means, deviations and products in FP64: n roundings of 2^-53 on sums of at most n - 1
    assert np.abs(got - ref).max() <= 8 * n * 2.0**-53
