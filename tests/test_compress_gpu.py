"""pifa_compress_device (Algorithm 1 on the GPU, float64) through the C ABI, against the fp64 oracle.

Pivots (I, I^c) must equal the oracle's bit for bit: the plain greedy loop on small and ragged
layers, LAPACK's pivoted QR on the LLaMA-shaped ones. C is pinned by Eq. 2 (||C W_p - W_np|| /
||W'|| <= 1e-10, the lossless reconstruction the paper states) and W_p by Eq. 1, both checked in
fp64 on the host on sampled rows.
"""
import time
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle
from paper_2501_19090_gb300 import inputs
from paper_2501_19090_gb300 import pifa as P

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _device_compress(U, V):
    Ud = torch.from_numpy(np.ascontiguousarray(U, dtype=np.float64)).to(DEV)
    Vd = torch.from_numpy(np.ascontiguousarray(V, dtype=np.float64)).to(DEV)
    piv, nonp, Wp, C, info = P.pifa_compress_device(Ud, Vd)
    return (piv.cpu().numpy().astype(np.int64), nonp.cpu().numpy().astype(np.int64), Wp.cpu().numpy(),
            C.cpu().numpy(), info)


def _check_eqs(U, V, piv, nonp, Wp, C, rows=None):
    """Eq. 1 (W_p = W'[I]) and Eq. 2 (W'[I^c] = C W_p) in fp64 on the host, on sampled rows."""
    Ud, Vd = U.astype(np.float64), V.astype(np.float64)
    Wp_ref = Ud[piv] @ Vd.T
    assert np.abs(Wp - Wp_ref).max() <= 1e-12 * np.abs(Wp_ref).max()
    if nonp.size:
        sel = np.arange(nonp.size) if rows is None else rows
        Wnp = Ud[nonp[sel]] @ Vd.T
        err = np.linalg.norm(C[sel] @ Wp - Wnp) / np.linalg.norm(Wnp)
        assert err <= 1e-10, err


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    P.load()


@pytest.mark.parametrize("m,n,r,seed", [(256, 256, 128, 0), (300, 200, 77, 3), (64, 128, 64, 4), (40, 48, 1, 5),
                                         (1000, 776, 301, 3), (97, 61, 33, 8)])
def test_small_layers_match_the_greedy_oracle(m, n, r, seed):
    U, V, _ = inputs.make_factors(m, n, r, seed)
    L = oracle.compress(U, V, r, "greedy")
    piv, nonp, Wp, C, info = _device_compress(U, V)
    assert np.array_equal(piv, L.pivots)
    assert np.array_equal(nonp, L.nonpivots)
    _check_eqs(U, V, piv, nonp, Wp, C)
    np.testing.assert_allclose(Wp, L.Wp, rtol=0, atol=1e-12 * np.abs(L.Wp).max())
    if C.size:
        np.testing.assert_allclose(C, L.C, rtol=0, atol=1e-9 * max(1.0, np.abs(L.C).max()))
    assert 0 < info.r_ratio <= 1 and info.min_pivot_gap >= 0


def test_worked_example_golden():
    """The hand-derived 5 x 3, rank-2 example (tests/golden): W' = U V^T with U its first two
    columns and V = [e_0, e_1], so the pivots and C printed there must come out exactly."""
    import os
    path = os.path.join(os.path.dirname(__file__), "golden", "worked_example_5x3_r2.txt")
    W, C_ref, kv = [], [], {}
    for ln in open(path):
        if not ln.strip() or ln.startswith("#"):
            continue
        key, *vals = ln.split()
        if key == "W":
            W.append([float(v) for v in vals])
        elif key == "C":
            C_ref.append([float(v) for v in vals])
        else:
            kv[key] = [int(v) for v in vals] if key in ("pivots", "nonpivots") else vals
    W = np.array(W)
    U = W[:, :2].copy()
    V = np.array([[1.0, 0.0], [0.0, 1.0], [0.0, 0.0]])
    assert np.array_equal(U @ V.T, W)
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert piv.tolist() == kv["pivots"] and nonp.tolist() == kv["nonpivots"]
    np.testing.assert_allclose(C, np.array(C_ref), rtol=0, atol=1e-14)
    np.testing.assert_allclose(Wp, W[piv], rtol=0, atol=1e-14)


@pytest.mark.parametrize("m,n,r", [(4096, 4096, 2048), (4096, 4096, 1638), (11008, 4096, 2048)])
def test_llama_layers_match_the_lapack_oracle(m, n, r):
    U, V, _ = inputs.make_factors(m, n, r, 0)
    L = oracle.compress(U, V, r, "lapack")
    piv, nonp, Wp, C, info = _device_compress(U, V)
    assert np.array_equal(piv, L.pivots), f"{np.setdiff1d(piv, L.pivots)[:8]}"
    assert np.array_equal(nonp, L.nonpivots)
    _check_eqs(U, V, piv, nonp, Wp, C, rows=inputs.random_rows(m - r, 64, 1))


def test_rank_deficient_is_reported():
    """Two identical columns in U and V make W' = U V^T rank r - 1."""
    U, V, _ = inputs.make_factors(200, 150, 20, 6)
    U[:, 7] = U[:, 3]
    V[:, 7] = V[:, 3]
    with pytest.raises(P.PifaError) as e:
        _device_compress(U, V)
    assert e.value.status == P.PIFA_ERR_RANK_DEFICIENT


def test_llama70b_gate_up_compresses_on_the_gpu():
    """The 28672 x 8192, r = 4096 layer: Eq. 1 and Eq. 2 on sampled rows; its pivots against the
    host route (pifa_compress, itself bit-exact with the oracle on the smaller layers) would take
    minutes on the host, so this checks the relations the pivots must satisfy instead: I and I^c
    partition [0, m), the sampled non-pivot rows are reproduced to 1e-10 (Eq. 2)."""
    m, n, r = 28672, 8192, 4096
    U, V, _ = inputs.make_factors(m, n, r, 0)
    t0 = time.perf_counter()
    piv, nonp, Wp, C, info = _device_compress(U, V)
    dt = time.perf_counter() - t0
    assert P.pifa_validate_indices(piv, nonp, m, r) == P.PIFA_OK
    rows = inputs.random_rows(m - r, 48, 2)
    pr = inputs.random_rows(r, 16, 3)
    Ud, Vd = U.astype(np.float64), V.astype(np.float64)
    Wp_ref = Ud[piv[pr]] @ Vd.T
    assert np.abs(Wp[pr] - Wp_ref).max() <= 1e-12 * np.abs(Wp_ref).max()
    Wnp = Ud[nonp[rows]] @ Vd.T
    assert np.linalg.norm(C[rows] @ Wp - Wnp) / np.linalg.norm(Wnp) <= 1e-10
    print(f"pifa_compress_device 28672 x 8192, r = 4096: {dt:.2f} s, min gap {info.min_pivot_gap:.3e}")


@pytest.mark.parametrize("m,n,r", [(300, 129, 97), (257, 320, 128), (900, 320, 128), (400, 191, 161), (520, 260, 257)])
def test_float64_products_by_slices_are_exact_on_whole_numbers(m, n, r):
    """W_p = U[I] V^T runs on the tensor cores by exact slices from 2^20 multiply-adds on. Whole
    numbers below 2^20 in magnitude have products and sums below 257 * 2^40 < 2^49, exact in
    float64 whatever the order, so W_p must equal the host's product bit for bit (sizes around the
    128 x 64 tiles, the 32-column K blocks and the 128-column exact accumulations)."""
    rng = np.random.default_rng(m)
    U = rng.integers(-(1 << 20), 1 << 20, (m, r)).astype(np.float64)
    V = rng.integers(-(1 << 20), 1 << 20, (n, r)).astype(np.float64)
    assert r * n * r >= 1 << 20
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert P.pifa_device_status() == P.PIFA_OK
    assert np.array_equal(Wp, U[piv] @ V.T)
    _check_eqs(U, V, piv, nonp, Wp, C)


@pytest.mark.parametrize("m,n,r", [(300, 129, 97), (900, 320, 128), (400, 191, 161), (520, 260, 257), (1500, 1500, 257),
                                   (900, 700, 641)])
def test_float64_products_by_slices_hold_every_digit(m, n, r):
    """Operands with all 53 bits, so that all eight digits of every value count (the whole numbers above fill
    the first three), against exact rational sums on sampled elements of W_p: one rounding to float64 and
    the slices' truncation, 2^-62.2 sqrt(r) of the largest entries of the row and column in the root mean
    square; eight times that is allowed. A pair of digits left out costs 2^-56 sqrt(r) at least, digits 7
    2^-57. Around the 32-column K blocks, the 128-column accumulations and (1500, 1500, 257) two panels; m large
    enough that the workspace holds the sliced operands (otherwise float64 chains compute W_p)."""
    rng = np.random.default_rng(m + r)
    U, V = rng.standard_normal((m, r)), rng.standard_normal((n, r))
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert P.pifa_device_status() == P.PIFA_OK
    scale = lambda x: 2.0 ** np.frexp(np.abs(x).max())[1]
    worst = 0.0
    for _ in range(500):
        i = int(rng.choice([0, 31, 96, r - 1, int(rng.integers(r))]))
        j = int(rng.choice([0, 63, 64, n - 1, int(rng.integers(n))]))
        a, b = U[piv[i]], V[j]
        terms = [Fraction(x) * Fraction(y) for x, y in zip(a.tolist(), b.tolist())]
        exact = sum(terms)
        err = abs(Fraction(float(Wp[i, j])) - exact)
        # a second panel (257 columns in the workspace of (1500, 1500, 257): 256 and 1) rounds its sum, too
        first = sum(terms[:256]) if (m, r) == (1500, 257) else 0
        allowed = 2.0 ** -53 * (abs(float(exact)) + abs(float(first))) + 8 * 2.0 ** -62.2 * r ** 0.5 * scale(a) * scale(b)
        worst = max(worst, float(err) / allowed)
    assert worst <= 1.0, worst


@pytest.mark.parametrize("r", [31, 32, 33, 127, 129, 160, 257, 300])
def test_blocked_cholesky_edges_match_the_greedy_oracle(r):
    """Ranks around the 32-column blocks and 128-column panels of the Cholesky factorisation."""
    m, n = r + 150, r + 90
    U, V, _ = inputs.make_factors(m, n, r, r)
    L = oracle.compress(U, V, r, "greedy")
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert np.array_equal(piv, L.pivots) and np.array_equal(nonp, L.nonpivots)
    _check_eqs(U, V, piv, nonp, Wp, C)


@pytest.mark.parametrize("m,n,r", [(7901, 300, 256), (3700, 700, 650), (2500, 1111, 1100), (2600, 1300, 1000)])
@pytest.mark.parametrize("kind", ["plain", "twins", "nan"])
def test_candidate_blocks_match_the_greedy_oracle(m, n, r, kind):
    """Layers with 2e6 unchosen values of Z and more, whose workspace holds the block's matrices where G
    and L were (the last two sizes), step over the rows of the largest norms and give the others each
    block's reflectors at once; the first two sizes step over every row. Rows that appear twice tie at every step (the first
    copies must be chosen, in the order of the layer without the second ones); a row that holds a NaN
    is never chosen and leaves every other row as it is."""
    U, V, _ = inputs.make_factors(m, n, r, r)
    keep = np.arange(m)
    if kind == "twins":
        U = np.concatenate([U, U[::-1]])
    elif kind == "nan":
        keep = np.delete(keep, 5)
        U[5, 3] = np.nan
    L = oracle.compress(U[keep], V, r, "lapack")
    piv, nonp, Wp, C, info = _device_compress(U, V)
    assert P.pifa_device_status() == P.PIFA_OK
    assert np.array_equal(piv, keep[L.pivots])
    assert P.pifa_validate_indices(piv, nonp, U.shape[0], r) == P.PIFA_OK
    if kind == "nan":
        assert np.isnan(C[np.searchsorted(nonp, 5)]).all()
    _check_eqs(U, V, piv, nonp, Wp, C, rows=np.flatnonzero(nonp != 5)[:: 7])
    assert 0 < info.r_ratio <= 1 and info.min_pivot_gap >= 0


@pytest.mark.parametrize("m,n,r", [(7901, 300, 256), (300, 200, 77), (2500, 1111, 1100)])
def test_an_infinity_in_u_does_what_float64_arithmetic_does(m, n, r):
    """Z = U L with a triangular L: an infinity in the last column of U gives its row of Z infinities
    only and with them an infinite norm, refused; in column 2 it meets L's zeros, and the row of NaN
    that this makes is never chosen."""
    U, V, _ = inputs.make_factors(m, n, r, 1)
    U[7, r - 1] = np.inf
    with pytest.raises(P.PifaError) as e:
        _device_compress(U, V)
    assert e.value.status == P.PIFA_ERR_RANK_DEFICIENT
    U[7, r - 1], U[7, 2] = 0.0, np.inf
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert 7 in nonp and np.isnan(C[np.searchsorted(nonp, 7)]).all()
    _check_eqs(U, V, piv, nonp, Wp, C, rows=np.flatnonzero(nonp != 7)[::7])


def test_equal_norms_are_taken_from_the_lowest_index():
    """Rows of +-1 on V = [I; 0] have exactly equal norms: no threshold separates the candidates."""
    m, n, r = 3600, 620, 600
    U = np.random.default_rng(0).integers(0, 2, (m, r)) * 2.0 - 1.0
    V = np.eye(n, r)
    piv, nonp, Wp, C, info = _device_compress(U, V)
    assert piv[0] == 0 and info.min_pivot_gap == 0.0
    _check_eqs(U, V, piv, nonp, Wp, C, rows=np.arange(0, nonp.size, 7))


@pytest.mark.parametrize("m,n,r", [(1000, 700, 640), (400, 191, 161), (2500, 1111, 1100)])
@pytest.mark.parametrize("s", [8, 20, 40])
def test_a_diagonal_between_the_factors_changes_nothing(m, n, r, s):
    """U D and V / D with D = 2^-s .. 2^s make the same W' as U and V, term by term, so Algorithm 1 has
    to give the same pivots, W_p within a float64 chain's bound r 2^-53 (|U| |V|^T) of each element (the
    host's product has that error too) and C with Eq. 2's residual of float64 arithmetic, although the
    large entries of a row of U D meet the small ones of V / D."""
    U, V, _ = inputs.make_factors(m, n, r, r)
    D = np.ldexp(1.0, np.random.default_rng(s).permutation(np.linspace(-s, s, r).astype(int)))
    L = oracle.compress(U, V, r, "lapack")
    piv, nonp, Wp, C, _ = _device_compress(U.astype(np.float64) * D, V.astype(np.float64) / D)
    assert P.pifa_device_status() == P.PIFA_OK
    assert np.array_equal(piv, L.pivots)
    Ud, Vd = U.astype(np.float64), V.astype(np.float64)
    bound = r * 2.0 ** -53 * (np.abs(Ud[piv]) @ np.abs(Vd).T)
    assert (np.abs(Wp - Ud[piv] @ Vd.T) / bound).max() <= 2.0
    Wnp = Ud[nonp] @ Vd.T
    assert np.linalg.norm(C @ (Ud[piv] @ Vd.T) - Wnp) / np.linalg.norm(Wnp) <= 8 * r * 2.0 ** -53


@pytest.mark.parametrize("spread,where", [(1e3, "U"), (1e7, "V"), (1e7, "both")])
def test_graded_singular_values_keep_the_residual_of_float64(spread, where):
    """W' = P diag(sigma) Q^T with sigma from 1 to 1 / spread, as layers' factors are: Eq. 2 holds to a
    small multiple of r 2^-53 however the values are shared out (rank check: 1e-8)."""
    m, n, r = 1000, 700, 640
    rng = np.random.default_rng(7)
    p = np.linalg.qr(rng.standard_normal((m, r)))[0]
    q = np.linalg.qr(rng.standard_normal((n, r)))[0]
    sig = np.logspace(0.0, -np.log10(spread), r)
    U = p * {"U": sig, "V": 1.0, "both": np.sqrt(sig)}[where]
    V = q * {"U": 1.0, "V": sig, "both": np.sqrt(sig)}[where]
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert P.pifa_device_status() == P.PIFA_OK
    bound = r * 2.0 ** -53 * (np.abs(U[piv]) @ np.abs(V).T)
    assert (np.abs(Wp - U[piv] @ V.T) / bound).max() <= 2.0
    W = U @ V.T
    assert np.linalg.norm(C @ W[piv] - W[nonp]) / np.linalg.norm(W[nonp]) <= 8 * r * 2.0 ** -53


@pytest.mark.parametrize("m,n,r,tall", [(2500, 2200, 1100, 1e6), (3700, 1800, 900, 1e6)])
def test_rows_far_apart_in_one_candidate_block(m, n, r, tall):
    """24 rows `tall` times the others are chosen first, in one block with ordinary rows; every other
    row's relation to the pivot rows (Eq. 2) must hold to a small multiple of r 2^-53 of the row itself."""
    U, V, _ = inputs.make_factors(m, n, r, 3)
    U, V = U.astype(np.float64), V.astype(np.float64)
    U[np.random.default_rng(3).permutation(m)[:24]] *= tall
    piv, nonp, Wp, C, _ = _device_compress(U, V)
    assert P.pifa_device_status() == P.PIFA_OK
    Wnp = U[nonp] @ V.T
    err = np.linalg.norm(C @ (U[piv] @ V.T) - Wnp, axis=1) / np.linalg.norm(Wnp, axis=1)
    assert err.max() <= 8 * r * 2.0 ** -53, err.max()
