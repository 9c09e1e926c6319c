"""The fixed-point kernels of the FP64 form against the oracle, at the edges of
their layouts and of their range.

Tolerance of moments within the spectral interval: 1e-12, a hundred times below the FP64
tolerance of the parity tests.  A component is rounded by at most 1/(2 U sqrt(D)) with
U > 2^52, so a step adds at most 2^-53 of the vector's norm, and n steps at most
n^2 2^-52 to mu_n: 5e-14 at n = 15 matrix-vector products."""
import ctypes

import numpy as np
import pytest
import torch

import kpm_workloads as W
import paper_2104_13218_gb300 as kpm
from oracle import c_oracle
from oracle import kpm_oracle as O

pytestmark = pytest.mark.gpu

K = 30


def _bonds(n, count):
    return W.random_bonds(n, count, 3, -0.7, 0.7)


def _check(model, n_up, R, a, b, tol=1e-12, **kw):
    got = kpm.moments(model, n_up, K, R, 5, a=[a] * len(n_up), b=[b] * len(n_up), **kw)
    bi, bj, J = model.arrays()
    for i, k in enumerate(n_up):
        ref = c_oracle.moments(model.n_sites, bi, bj, J, k, a, b, K, R, 5)
        for q in ref:
            err = np.abs(got[q][i] - ref[q]) / np.maximum(1.0, np.abs(ref[q]))
            assert err.max() <= tol, (k, q, err.max())
    return got


# rows of 2 .. 64 chunks: one lane pair, odd and even numbers of chunks, both sides
# of one chunk per lane and the largest that uses the lists
@pytest.mark.parametrize("R", [3, 4, 5, 8, 25, 31, 32, 33, 63, 64, 65, 100, 127, 128])
def test_row_layouts(R):
    _check(W.j1j2_chain(10, 1.0, 0.4), [0, 1, 5, 7, -1], R, 6.0, -1.0)


# one to four coupling groups, ferromagnetic and zero couplings, an empty sector list's
# neighbours (one state), and the largest group the lists take (lowest unit)
def test_couplings():
    n = 9
    for groups in ((1.0,), (1.0, -0.5), (1.0, -0.5, 0.25), (1.0, 0.0, 0.25, -2.0)):
        bonds = [(i, (i + 1 + d) % n, J) for d, J in enumerate(groups) for i in range(n)]
        model = W._model("groups", n, bonds)
        _check(model, [0, 1, 4, -1], 6, 12.0, -1.0)
    full = W._model("complete22", 22, [(i, j, 1.0) for i in range(22) for j in range(i)])
    _check(full, [0, 1, 2, 22], 6, 70.0, -10.0)


# the interval may end at the spectrum (eps = 0): coefficients of exactly 2
def test_band_edge_coefficients():
    model = W.ring(8)
    _check(model, [0, 2, 4], 7, 3.0, -1.0)


# a spectrum outside [-1, 1]: the moments grow beyond the fixed-point range and
# the run is made with FP64 vectors, status KPM_EBOUNDS
@pytest.mark.parametrize("a", [1.2, 0.4, 1e-3])
def test_spectrum_outside_the_interval(a):
    model = W.ring(12)
    n_up = [4, 6, -1]
    got = kpm.moments(model, n_up, K, 9, 5, a=[a] * 3, b=[-1.0] * 3, allow_ebounds=True)
    assert got["status"] == 6
    bi, bj, J = model.arrays()
    for i, k in enumerate(n_up):
        ref = c_oracle.moments(12, bi, bj, J, k, a, -1.0, K, 9, 5)
        for q in ref:
            scale = np.abs(ref[q]) + np.abs(ref["mu"]).max() * 1e-12
            assert (np.abs(got[q][i] - ref[q]) <= 1e-9 * scale).all(), (k, q)


def test_per_vector_moments():
    model = W.ladder(10)
    n_up, R = [3, 5], 37
    got = kpm.moments(model, n_up, K, R, 5, a=[9.0] * 2, b=[-2.0] * 2, per_vector=True)
    bi, bj, J = model.arrays()
    for i, k in enumerate(n_up):
        for r in (0, 17, R - 1):
            ref = c_oracle.moments(10, bi, bj, J, k, 9.0, -2.0, K, 1, 5, r)["mu"]
            assert np.abs(got["mu_r"][i, r] - ref).max() <= 1e-12
        assert np.abs(got["mu_r"][i].mean(0) - got["mu"][i]).max() <= 1e-13


# ---------------------------------------------------------------- scratch
# nothing may depend on what the scratch held before: workspaces filled with NaN
# bit patterns (one list run, lists with matrix elements, small sectors, one-lane
# rows, both precisions, and the reverse sweep of both layouts)

def _dirty(size):
    return torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("R", [2, 4, 25, 33, 64])
def test_moments_in_a_used_workspace(R, precision):
    for model, n_up in ((W.j1j2_chain(15, 1.0, 0.4), [7, 5]), (_bonds(15, 37), [7]), (W.ring(15), [-1]),
                        (W.ladder(8), [4, 8])):
        S = len(n_up)
        kw = dict(a=[15.0] * S, b=[0.0] * S, precision=precision, device=True)
        ws = _dirty(kpm.moments_workspace_size(model, n_up, 12, R, precision))
        ref = kpm.moments(model, n_up, 12, R, 5, **kw)
        got = kpm.moments(model, n_up, 12, R, 5, workspace=ws, **kw)
        for q in ("mu", "mu_M", "mu_M2"):
            assert torch.equal(got[q], ref[q]), (model.name, q)
        bi, bj, J = model.arrays()
        mu = c_oracle.moments(model.n_sites, bi, bj, J, n_up[0], 15.0, 0.0, 12, R, 5)["mu"]
        assert np.abs(got["mu"][0].cpu().numpy() - mu).max() <= (1e-12 if precision == "fp64" else 1e-5)


@pytest.mark.parametrize("R", [3, 4, 25, 32, 33, 65])
def test_gradient_in_a_used_workspace(R):
    for model in (W.j1j2_chain(9, 1.0, 0.35), _bonds(9, 17)):
        g = {"mu": np.random.default_rng(3).standard_normal((2, 12))}
        P = int(model.classes().max()) + 1
        args = (model, model.classes(), P, [4, 6], [8.0] * 2, [-1.0] * 2, 12, R, 17, g)
        ws = _dirty(kpm.moments_backward_workspace_size(model, [4, 6], 12, R))
        got = kpm.moments_backward(*args, workspace=ws)
        bi, bj, J = model.arrays()
        ref = sum(O.moment_jacobian(9, bi, bj, J, model.classes(), k, 8.0, -1.0, 12, R, 17) @ g["mu"][i]
                  for i, k in enumerate((4, 6)))
        assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()


# ---------------------------------------------------------------- reverse sweep
# against the oracle's tangents, with the parity tests' relative tolerance (1e-9
# of the sum of |d mu / d theta| |cotangent|)

def _gradient(R, K, scale, a=6.0, n_up=(4, 5, 7), on_zero=None, ckpt=0):
    model = W.j1j2_chain(10, 1.0, 0.35)
    bi, bj, J = model.arrays()
    n_up, S = list(n_up), len(n_up)
    g = {q: np.random.default_rng(3).standard_normal((S, K)) * scale for q in ("mu", "mu_M", "mu_M2")}
    if on_zero is not None:
        for q in g:
            g[q][on_zero] = 0.0
    got = kpm.moments_backward(model, model.classes(), 2, n_up, [a] * S, [-1.0] * S, K, R, 17, g,
                               ckpt_interval=ckpt)
    ref, size = np.zeros(2), np.zeros(2)
    for i, k in enumerate(n_up):
        jac = O.moment_jacobian(10, bi, bj, J, model.classes(), k, a, -1.0, K, R, 17)
        w = g["mu"][i] + (k - 5) * g["mu_M"][i] + (k - 5) ** 2 * g["mu_M2"][i]
        ref += jac @ w
        size += np.abs(jac) @ np.abs(w)
    return got, ref, size


@pytest.mark.parametrize("R", [3, 4, 25, 32, 33, 64, 65, 128])
def test_gradient_layouts(R):
    got, ref, size = _gradient(R, 24, 1.0)
    assert (np.abs(got - ref) <= 1e-9 * size).all(), (got, ref)


# the shortest runs; cotangents of extreme size, growing and falling with the
# order by many powers of two per step, and zero for one sector
@pytest.mark.parametrize("K", [2, 4, 40])
@pytest.mark.parametrize("scale", ["one", "tiny", "huge", "growing", "falling"])
def test_gradient_scales(K, scale):
    n = np.arange(K)
    f = {"one": np.ones(K), "tiny": np.full(K, 1e-200), "huge": np.full(K, 1e200),
         "growing": 10.0 ** n, "falling": 10.0 ** -n}[scale]
    got, ref, size = _gradient(8, K, f, on_zero=1)
    assert (np.abs(got - ref) <= 1e-9 * size).all(), (got, ref)


def test_gradient_of_zero_and_of_nan():
    got, _, _ = _gradient(8, 12, 0.0)
    assert (got == 0.0).all()
    got, _, _ = _gradient(8, 12, np.where(np.arange(12) == 5, np.nan, 1.0))
    assert np.isnan(got).all()


# vectors that leave the range: the sweep is made in FP64 (which regenerates growing
# vectors from stored pairs: two steps apart at most)
def test_gradient_outside_the_interval():
    got, ref, size = _gradient(8, 24, 1.0, a=1.0, ckpt=2)
    assert (np.abs(got - ref) <= 1e-9 * size).all(), (got, ref)


# ---------------------------------------------------------------- lists with matrix elements
# couplings of more values than groups: fixed point (tolerance as above) and FP32
# (the parity tests' 1e-5); rows of one and two chunks per lane

@pytest.mark.parametrize("R", [3, 4, 25, 32, 64, 65, 128])
def test_many_couplings(R):
    _check(_bonds(10, 23), [0, 1, 5, 8, -1], R, 9.0, 0.5)


@pytest.mark.parametrize("R", [5, 50, 128, 132, 256])
def test_many_couplings_fp32(R):
    _check(_bonds(12, 30), [6, 8, -1], R, 9.0, 0.5, 1e-5, precision="fp32")


# the most bonds, and a number of neighbours at and next to whole batches
@pytest.mark.parametrize("count", [5, 6, 7, 8, 253])
def test_list_lengths(count):
    model = _bonds(23 if count > 100 else 8, count)
    _check(model, [1, 2], 6, 45.0 if count > 100 else 6.0, 0.0)


@pytest.mark.parametrize("a", [2.0, 1e-3])
def test_many_couplings_outside_the_interval(a):
    model = _bonds(10, 23)
    got = kpm.moments(model, [5], K, 9, 5, a=[a], b=[0.5], allow_ebounds=True)
    assert got["status"] == 6
    bi, bj, J = model.arrays()
    ref = c_oracle.moments(10, bi, bj, J, 5, a, 0.5, K, 9, 5)["mu"]
    assert (np.abs(got["mu"][0] - ref) <= 1e-9 * (np.abs(ref) + 1e-12 * np.abs(ref).max())).all()


def _check_spin(two_s, n, Q, R, a, b, tol, precision):
    model = W.j1j2_chain(n, 1.0, -0.4)
    got = kpm.spin_moments(model, two_s, Q, K, R, 5, [a] * len(Q), [b] * len(Q), precision=precision,
                           allow_ebounds=True)
    bi, bj, J = model.arrays()
    for i, q in enumerate(Q):
        ref = c_oracle.spin_moments(n, two_s, bi, bj, J, q, a, b, K, R, 5)
        for k in ref:
            err = np.abs(got[k][i] - ref[k]) / np.maximum(np.maximum(1.0, np.abs(ref[k])),
                                                           1e-12 * np.abs(ref["mu"]).max())
            assert err.max() <= tol, (q, k, err.max())
    return got


@pytest.mark.parametrize("R", [1, 2, 3, 16, 33, 128, 129])
def test_spin_lists(R):
    for two_s, n, a in ((1, 8, 7.0), (2, 5, 12.0), (7, 4, 70.0)):
        top = two_s * n
        _check_spin(two_s, n, [0, 1, top // 2, -1], R, a, 0.0, 1e-12, "fp64")


@pytest.mark.parametrize("R", [1, 4, 20, 128, 132, 257])
def test_spin_lists_fp32(R):
    _check_spin(3, 5, [7, -1], R, 28.0, 0.0, 1e-5, "fp32")


def test_spin_outside_the_interval():
    got = _check_spin(3, 5, [7, -1], 5, 2.0, 0.0, 1e-9, "fp64")
    assert got["status"] == 6


# ---------------------------------------------------------------- small sectors in one launch
# any number of vectors, sectors of 1 state to the largest that fits, more and
# fewer blocks than SMs; groups and bonds with their own couplings; whole space

@pytest.mark.parametrize("R", [1, 2, 7, 40, 200])
def test_small_sectors(R):
    _check(W.ladder(10), list(range(11)), R, 9.0, -2.0)
    _check(_bonds(9, 17), [0, 4, 9, -1], R, 7.0, 0.0)


def test_largest_small_sector_and_the_next():
    model = W.j1j2_chain(16, 1.0, 0.4)  # 12870 states
    _check(model, [8, 7, 1], 2, 9.0, -1.5)
    _check(_bonds(16, 40), [8], 1, 15.0, 0.0)
    _check(W.ring(13), [-1], 2, 4.8, -1.2)  # 2^13
    _check(W.ring(14), [-1], 2, 5.2, -1.4)  # 2^14: the list kernels


# 256 equal bonds between two sites: a count that 8 bits do not hold
def test_more_bonds_than_a_byte_counts():
    model = W._model("many", 3, [(0, 1, 0.01)] * 256)
    _check(model, [0, 1, 2, -1], 5, 3.0, 0.0)


def test_small_sectors_single_product():
    model = W.ring(6)
    got = kpm.moments(model, [3, 2], 2, 3, 5, a=[2.4] * 2, b=[-0.6] * 2)
    bi, bj, J = model.arrays()
    for i, k in enumerate((3, 2)):
        ref = c_oracle.moments(6, bi, bj, J, k, 2.4, -0.6, 2, 3, 5)["mu"]
        assert np.abs(got["mu"][i] - ref).max() <= 1e-14


# ---------------------------------------------------------------- M-weighted sums of the whole space
# With -J and -b in place of J and b every v_n becomes (-1)^n v_n, bit for bit, so
# the odd moments change sign and nothing else: what is left of their sum is a bias of the sums.
# Tolerance: four roundings of a double in [0.5, 1).  Units near the lowest, rows with
# unused columns; lists with matrix elements, with groups, and small sectors.
@pytest.mark.parametrize("n,count,R", [(17, 100, 3), (17, -48, 5), (12, 60, 3)])
def test_weighted_sums_have_no_bias(n, count, R):
    bi, bj, J = _bonds(n, abs(count)).arrays()
    J = J if count > 0 else np.ones_like(J)
    got = [kpm.moments(kpm.CModel(n, bi, bj, s * J), [-1], 12, R, 5, a=[30.0], b=[0.5 * s]) for s in (1, -1)]
    for q in ("mu", "mu_M", "mu_M2"):
        assert np.abs(got[0][q][0, 1::2] + got[1][q][0, 1::2]).max() <= 4.5e-16, q
        assert np.abs(got[0][q][0, 0::2] - got[1][q][0, 0::2]).max() <= 4.5e-16, q


# ---------------------------------------------------------------- coefficients
# Against the recursion in extended precision with the same a and b (80 or 128 bits).  A level
# of H' that is off by d moves mu_n by up to n d.  Coefficients are rounded to 2^-60: with 8
# (spin 5/2: 4) bonds d <= 9 2^-60 (diagonal and flips: twice), at n = 1000 so 1.6e-14; the
# vectors' roundings of 0.29/U in the mean square add 4 sqrt(n sum U_k^2) 0.29/(U sqrt(DR)),
# below 4e-15 at D R = 768 for a mean square of 10 of the U_k, five sigma; sums 1e-15.
def _extended(codes, diag, rows, cols, vals, a, b, K, R, seed, M):
    L = np.longdouble
    mask = (1 << 64) - 1

    def sm(x):
        z = (x + 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    h = [sm(sm(seed) ^ r) for r in range(R)]
    x = np.array([[-1 if sm(hr ^ int(c)) >> 63 else 1 for hr in h] for c in codes]).astype(L)
    a, b = L(a), L(b)
    order = np.argsort(rows, kind="stable")
    rows, cols, vals = rows[order], cols[order], vals[order][:, None]
    starts = np.searchsorted(rows, np.arange(len(codes)))
    has = np.bincount(rows, minlength=len(codes)) > 0

    def hp(v):
        off = np.zeros_like(v)
        off[has] = np.add.reduceat(vals * v[cols], starts[has], axis=0)
        return ((diag[:, None] - b) * v + off) / a

    def dots(y):
        return [np.array([(w * (u * y).sum(1)).sum() for w in (1, M, M * M)]) / (L(len(codes)) * R) for u in (x,)][0]

    y = hp(x)
    d = [dots(x), None]
    d[1] = dots(y)
    f0, f1 = d
    for _ in range(1, K // 2):
        x, y = y, 2 * hp(y) - x
        d += [2 * dots(x) - f0, 2 * dots(y) - f1]
    return np.array(d).T


def test_coefficients_small_sectors():
    n, J, a, b, K, R = 8, 1.0073, 3.0917, -0.8931, 2000, 3
    L = np.longdouble
    codes = np.arange(1 << n)
    diag, rows, cols = np.zeros(1 << n, L), [], []
    for i in range(n):
        m = (1 << i) | (1 << (i + 1) % n)
        anti = ((codes & m) != 0) & ((codes & m) != m)
        diag += L(J) * np.where(anti, L(-0.25), L(0.25))
        rows.append(codes[anti])
        cols.append(codes[anti] ^ m)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    M = np.array([bin(c).count("1") - n / 2 for c in codes]).astype(L)
    ref = _extended(codes, diag, rows, cols, np.full(len(rows), L(J) / 2), a, b, K, R, 5, M)
    got = kpm.moments(W.ring(n, J), [-1], K, R, 5, a=[a], b=[b])
    for i, q in enumerate(("mu", "mu_M", "mu_M2")):
        assert np.abs(got[q][0] - ref[i]).max() <= 2.2e-14 * (1, 1.5, n / 4)[i], q


def test_coefficients_spin():
    n, two_s, J, a, b, K, R = 4, 5, 1.0073, 28.1237, -2.4931, 2000, 1
    L = np.longdouble
    d = two_s + 1
    rank = np.arange(d ** n)
    q = np.stack([(rank // d ** i) % d for i in range(n)])
    codes = sum(q[i].astype(np.int64) << (3 * i) for i in range(n))
    where = {int(c): k for k, c in enumerate(codes)}
    m2 = 2 * q - two_s
    diag, rows, cols, vals = np.zeros(len(rank), L), [], [], []
    for i in range(n):
        j = (i + 1) % n
        diag += L(J) / 4 * (m2[i] * m2[j])
        for s in (1, -1):
            p, r = (i, j) if s == 1 else (j, i)
            k = (two_s - q[p]) * (q[p] + 1) * q[r] * (two_s - q[r] + 1)
            ok = k > 0
            rows.append(rank[ok])
            cols.append(np.array([where[int(c)] for c in codes[ok] + (1 << 3 * p) - (1 << 3 * r)]))
            vals.append(L(J) / 2 * np.sqrt(k[ok].astype(L)))
    ref = _extended(codes, diag, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), a, b, K, R,
                    5, m2.sum(0).astype(L) / 2)
    got = kpm.spin_moments(W.ring(n, J), two_s, [-1], K, R, 5, [a], [b])
    for i, (k, scale) in enumerate((("mu", 1), ("mu_M", 3.5), ("mu_M2", 12))):
        assert np.abs(got[k][0] - ref[i]).max() <= 2.2e-14 * scale, k


# ---------------------------------------------------------------- dot products of FP32 spin runs
# They are sums of exact products as if in FP64.  All components of v_0 are +-x, so mu_0 is
# D x^2; tolerance: 30 roundings of FP64 (the sum over a tile's lanes, the tiles and the vectors).
@pytest.mark.parametrize("two_s,n,Q,R", [(2, 12, 12, 100), (5, 8, 20, 60), (5, 5, 12, 4)])
def test_dot_products_of_fp32_spin_runs(two_s, n, Q, R):
    D = kpm.lib().kpm_spin_sector_dim(n, two_s, Q)
    got = kpm.spin_moments(W.ring(n), two_s, [Q], 2, R, 5, [90.0], [0.0], precision="fp32")
    x = float(np.float32(1.0 / np.sqrt(float(D))))
    assert abs(got["mu"][0, 0] - D * x * x) <= 30 * 2.0 ** -53


def _step_launches(call):
    """Device time (ms) and number of the step launches that a call makes."""
    ms, n = ctypes.c_double(), ctypes.c_int64()
    kpm.lib().kpm_profile_enable(1)
    call()
    kpm.lib().kpm_profile_read(ctypes.byref(ms), ctypes.byref(n), None)
    kpm.lib().kpm_profile_enable(0)
    return ms.value, n.value


# A run that leaves the range in its first ten steps or so (levels of H' down to -1.6) does not pay for the others: its step launches
# take no longer than those of the FP64 run that replaces it (unit vectors are run in FP64) and a
# part of a fixed-point run's.
def test_abandoned_run_stops():
    def step_ms(a, **kw):
        for _ in range(2):
            r = _step_launches(lambda: kpm.moments(W.ring(20), [10], 200, 20, 5, a=[a], b=[-1.0],
                                                   allow_ebounds=True, device=True, **kw))
        return r

    fixed, fp64, left = step_ms(30.0), step_ms(30.0, vectors="basis"), step_ms(5.0)
    assert left[1] == fixed[1] + fp64[1] and fp64[0] > 2 * fixed[0]
    assert left[0] < fp64[0] + 0.5 * fixed[0], (fixed, fp64, left)


# The launch that makes all products of small sectors is among the recorded step launches.
def test_small_sector_launch_is_recorded():
    ms, n = _step_launches(lambda: kpm.moments(W.ring(12), [6], 200, 20, 5, a=[5.0], b=[-1.0]))
    assert n == 1 and ms > 0.0


# ---------------------------------------------------------------- sums of many tiles, runs of parts

# sectors of more tiles than one block sums, with groups and with couplings of their own
@pytest.mark.parametrize("model", [W.j1j2_chain(20, 1.0, 0.4), W.random_bonds(20, 30, 3, -0.7, 0.7)],
                         ids=lambda m: m.name)
def test_sums_in_several_parts(model):
    bi, bj, J = model.arrays()
    got = kpm.moments(model, [10], 8, 100, 5, a=[15.0], b=[0.5])
    # (the oracle adds one product after the other: over all vectors at once it is itself off
    # by 2.2e-12, mu_0 = 1 - 2.2e-12)
    ref = np.mean([c_oracle.moments(20, bi, bj, J, 10, 15.0, 0.5, 8, 5, 5, r0)["mu"]
                   for r0 in range(0, 100, 5)], axis=0)
    assert np.abs(got["mu"][0] - ref).max() <= 1e-12


# a shorter run's moments are the first of a longer run's, bit for bit
@pytest.mark.parametrize("model,n_up,R", [(W.ladder(12), [6, 7], 20), (W.j1j2_chain(20, 1.0, 0.4), [10], 100),
                                          (W.random_bonds(18, 30, 3, -0.7, 0.7), [9, 5], 20), (W.ring(17), [-1], 9)])
def test_shorter_runs_are_prefixes(model, n_up, R):
    kw = dict(a=[16.0] * len(n_up), b=[0.5] * len(n_up), device=True)
    short, long_ = (kpm.moments(model, n_up, K, R, 5, **kw) for K in (12, 24))
    for q in ("mu", "mu_M", "mu_M2"):
        assert torch.equal(short[q], long_[q][:, :12]), q


# FP32 with a large sector, and a small one (in FP64) whose interval is too narrow: both runs are
# made again, on two streams
def test_fp32_side_run_outside_the_interval():
    model, n_up, a, b = W.ring(16), [8, 2], [6.0, 1.0], [-1.0, 3.0]
    got = kpm.moments(model, n_up, K, 20, 5, a=a, b=b, precision="fp32", allow_ebounds=True)
    assert got["status"] == 6
    bi, bj, J = model.arrays()
    refs = [c_oracle.moments(16, bi, bj, J, k, a[i], b[i], K, 20, 5)["mu"] for i, k in enumerate(n_up)]
    assert np.abs(got["mu"][0] - refs[0]).max() <= 1e-5
    scale = np.abs(refs[1]) + 1e-12 * np.abs(refs[1]).max()
    assert (np.abs(got["mu"][1] - refs[1]) <= 1e-9 * scale).all()


# A sector of one state has the moments cos(n arccos x), x = (E - b)/a, without an average over
# states: an x that is off by d moves mu_n by n d / sqrt(1 - x^2).  x is rounded to 2^-60; the vector's
# roundings of 0.29/U in the root mean square (U = 2^54 - 1 for 9 bonds) add up to 1.2 sqrt(n) times
# that after n products, and mu_2n = 2 v_n^2 - 1 to four times that (six standard deviations).
def test_sector_of_one_state():
    n, J, a, b, K = 9, 1.0077, 3.0917, 0.5931, 800
    got = kpm.moments(W.ring(n, J), [n], K, 3, 5, a=[a], b=[b])["mu"][0]
    L = np.longdouble
    x = (L(J) * n / 4 - L(b)) / L(a)
    assert 1 / np.sqrt(1 - x * x) < 1.2
    t = [L(1), x]
    for _ in range(K - 2):
        t.append(2 * x * t[-1] - t[-2])
    tol = 1.2 * K * 2.0 ** -60 + 6 * 4 * 1.2 * np.sqrt(K / 2) * 0.29 * 2.0 ** -54
    assert np.abs(got - np.array(t)).max() <= tol


# The even moments have no common offset: 2 <v_n|v_n> - <v_0|v_0> is formed before it is rounded
# (rounded by itself, <v_0|v_0> leaves up to 1e-16, the same for all vectors).  The vectors' own
# roundings move mu_2n by 4 sqrt(n) 0.29/(U sqrt(D R)), 1.3e-17 at most here (U > 2^53, D R > 2000), and
# their mean over 29 moments by a fifth of that; six standard deviations.
@pytest.mark.parametrize("Q,R", [(8, 7), (9, 5), (10, 4), (11, 6), (12, 3), (13, 5)])
def test_even_moments_have_no_offset(Q, R):
    n, two_s, J, a, b, K = 5, 5, 1.0073, 40.1237, -6.4931, 60
    L = np.longdouble
    rank = np.arange(6 ** n)
    q = np.stack([(rank // 6 ** i) % 6 for i in range(n)])
    codes = sum(q[i].astype(np.int64) << (3 * i) for i in range(n))
    order = np.argsort(codes)
    order = order[q.sum(0)[order] == Q]
    codes, q = codes[order], q[:, order]
    where = {int(c): k for k, c in enumerate(codes)}
    diag, rows, cols, vals = np.zeros(len(codes), L), [], [], []
    for i in range(n):
        j = (i + 1) % n
        diag += L(J) / 4 * ((2 * q[i] - two_s) * (2 * q[j] - two_s))
        for p, r in ((i, j), (j, i)):
            k = (two_s - q[p]) * (q[p] + 1) * q[r] * (two_s - q[r] + 1)
            ok = np.nonzero(k > 0)[0]
            rows.append(ok)
            cols.append(np.array([where[int(c)] for c in codes[ok] + (1 << 3 * p) - (1 << 3 * r)]))
            vals.append(L(J) / 2 * np.sqrt(k[ok].astype(L)))
    ref = _extended(codes, diag, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), a, b, K, R, 5,
                    np.zeros(len(codes), L))[0]
    got = kpm.spin_moments(W.ring(n, J), two_s, [Q], K, R, 5, [a], [b])["mu"][0]
    assert len(codes) * R > 2000 and abs((got - ref)[2::2].mean()) <= 6 * 1.3e-17 / 5


# Coefficients within the range and levels outside [-1, 1]: the components leave the range during
# the run, which is given up and made again in FP64 (small sectors and whole space, lists,
# bonds of their own in both; gradient and spin s below).
@pytest.mark.parametrize("model,n_up,R,a", [
    (W.ring(12), [4, 6, -1], 9, 3.6), (W.ring(16), [8], 9, 4.8), (W.ring(17), [-1], 5, 5.1), (_bonds(10, 23), [5, -1], 9, 1.6),
    (_bonds(17, 34), [8], 9, 2.4)], ids=lambda v: getattr(v, "name", None))
def test_components_leave_the_range(model, n_up, R, a):
    bi, bj, J = model.arrays()
    b = 0.0 if model.name.startswith("ring") else 0.25 * float(np.sum(J))
    got = kpm.moments(model, n_up, K, R, 5, a=[a] * len(n_up), b=[b] * len(n_up), allow_ebounds=True)
    assert got["status"] == 6
    for i, k in enumerate(n_up):
        ref = c_oracle.moments(model.n_sites, bi, bj, J, k, a, b, K, R, 5)
        for q in ref:
            scale = np.abs(ref[q]) + np.abs(ref[q]).max() * 1e-12
            assert (np.abs(got[q][i] - ref[q]) <= 1e-9 * scale).all(), (k, q)


def test_gradient_components_leave_the_range():
    got, ref, size = _gradient(8, 40, 1.0, a=3.5, ckpt=2)
    assert (np.abs(got - ref) <= 1e-9 * size).all(), (got, ref)


def test_spin_components_leave_the_range():
    got = _check_spin(3, 5, [7, -1], 5, 6.0, 0.0, 1e-9, "fp64")
    assert got["status"] == 6
