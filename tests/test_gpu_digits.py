"""FP64 products from exact integer digit products (csrc/digits.cu): the sizes
where tiles, stages, blocks and chunks end, strides, scales, and what cannot
be split."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ttsn():
    import torch

    assert torch.cuda.is_available()
    import paper_2503_18056_gb300 as m

    return m


def _call(ttsn, A, B, ta, tb, alpha=1.0, pad=0):
    """tt_dgemm with leading dimensions `pad` wider than the matrices."""
    import torch

    from paper_2503_18056_gb300 import _native

    def dev(X):
        P = torch.full((X.shape[0], X.shape[1] + pad), float("nan"), dtype=torch.float64, device="cuda")
        P[:, : X.shape[1]] = torch.as_tensor(X)
        return P

    M, K = A.shape[::-1] if ta else A.shape
    N = B.shape[0] if tb else B.shape[1]
    a, b = dev(A), dev(B)
    c = torch.full((M, N + pad), -7.0, dtype=torch.float64, device="cuda")
    st = _native.lib.tt_dgemm(int(ta), int(tb), M, N, K, alpha, ctypes.c_void_p(a.data_ptr()), a.shape[1],
                              ctypes.c_void_p(b.data_ptr()), b.shape[1], 0.0, ctypes.c_void_p(c.data_ptr()),
                              c.shape[1], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    assert bool((c[:, N:] == -7.0).all())
    return c[:, :N].cpu().numpy()


# (M, N, K): one past and one short of the 128 x 64 tile, the 32-index stage,
# the 512-index block, the row forms' 64 / 128 / 256 / 512 / 1024 entries, and
# a contraction long enough for several splits
SIZES = [(500, 500, 64), (129, 1999, 65), (1023, 63, 257), (127, 257, 513), (511, 33, 1024), (385, 65, 1025),
         (32, 16, 40001), (2003, 17, 601)]


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
def test_integer_products_are_exact(ttsn, M, N, K, ta, tb):
    # entries of 18 bits: every sum is an integer below 2^53, so the FP64
    # product is exact too and any lost digit, row or index shows
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-(1 << 17), 1 << 17, (K, M) if ta else (M, K)).astype(float)
    B = rng.integers(-(1 << 17), 1 << 17, (N, K) if tb else (K, N)).astype(float)
    ref = (A.T if ta else A).astype(np.int64) @ (B.T if tb else B).astype(np.int64)
    assert np.array_equal(_call(ttsn, A, B, ta, tb, pad=3), ref.astype(float))


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("grade", [0, 8])
def test_split_error_is_within_its_bound(ttsn, M, N, K, grade):
    """Rows graded over 8 decades along and across the contraction.  A term
    loses the levels s + t >= 8 (at most 7.1 * 2^12 * 128^-10 of 2^(e_i + e_j),
    which is at most 16 max|a_i| max|b_j|) and the 56-bit rounding of both
    factors (2 * 2^-57 of 4 max|a_i| max|b_j|): together under 2^-51; the FP64
    reference is off by K eps sum |a||b| at most."""
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    if grade:
        A *= 10.0 ** (-grade * rng.random(K))[None, :] * 10.0 ** (grade * rng.random(M))[:, None]
        B *= 10.0 ** (-grade * rng.random(N))[:, None]
    ref = A @ B.T
    got = _call(ttsn, A, B, False, True, alpha=1.0)
    bound = K * 2.0 ** -51 * np.abs(A).max(1)[:, None] * np.abs(B).max(1)[None, :] \
        + (K + 1) * np.finfo(float).eps * (np.abs(A) @ np.abs(B).T)
    assert np.all(np.abs(got - ref) <= bound)
    # alpha scales the rounded result once more
    scaled = _call(ttsn, A, B, False, True, alpha=-0.75)
    assert np.array_equal(scaled, -0.75 * got)


@pytest.mark.parametrize("m,n", [(1025, 130), (40001, 33), (9001, 129), (140000, 65), (20000, 449)])
def test_gram_integer_products_are_exact_and_symmetric(ttsn, m, n):
    import torch

    rng = np.random.default_rng(m)
    A = rng.integers(-(1 << 16), 1 << 16, (m, n)).astype(float)
    G = ttsn.gram(torch.as_tensor(A, device="cuda")).cpu().numpy()
    ref = A.astype(np.int64).T @ A.astype(np.int64)
    assert np.array_equal(G, ref.astype(float)) and np.array_equal(G, G.T)


def test_inf_nan_and_extreme_scales_take_the_fp64_pipe(ttsn):
    rng = np.random.default_rng(0)
    A, B = rng.standard_normal((300, 260)), rng.standard_normal((260, 310))
    for a, b in ((np.inf, 1.0), (1.0, np.nan), (-np.inf, np.inf)):
        X, Y = A.copy(), B.copy()
        X[5, 7] *= a
        Y[11, 9] *= b
        with np.errstate(all="ignore"):
            ref = X @ Y
        got = _call(ttsn, X, Y, False, False)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
        fine = np.isfinite(ref)
        assert np.abs(got[fine] - ref[fine]).max() <= 1e-13 * np.abs(ref[fine]).max() * np.sqrt(260)
    for sa, sb in ((1e-290, 1e280), (1e-310, 1e300), (0.0, 1.0)):
        ref = (sa * A) @ (sb * B)
        got = _call(ttsn, sa * A, sb * B, False, False)
        assert np.abs(got - ref).max() <= 1e-13 * max(np.abs(ref).max(), 1e-300) * np.sqrt(260)


def test_captured_steps_above_the_digit_sizes_equal_host_steps(ttsn):
    """A grid whose grown-core products take the digit form: a captured step
    decides it from the device's sizes and gives the host-driven bits."""
    import torch

    import workloads

    p = workloads.problem("small_2d", n=(96, 90), n_theta=16, n_phi=32, eps=1e-6, bc=1)
    p["max_rank"] = 24
    a, b = ttsn.TTSN.from_problem(p), ttsn.TTSN.from_problem(p)
    b.set_graph(True)
    for _ in range(5):
        assert a.step()["ranks"] == b.step()["ranks"]
    assert 96 * 90 * (5 * a.ranks()[1] + 1) ** 2 > 16e6
    assert torch.equal(a.full(), b.full())


@pytest.mark.parametrize("M,N,K", [(300, 260, 260), (2100, 1100, 1100), (260, 300, 2000)])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
def test_small_entries_that_meet_large_ones_keep_their_accuracy(ttsn, M, N, K, ta, tb):
    """A @ (a selection of columns) gives A's entries, whatever their range in a
    row: the sums hold one term, so nothing is rounded."""
    rng = np.random.default_rng(K)
    A = rng.standard_normal((M, K)) * 10.0 ** (-40 * rng.random((M, K)))
    pick = rng.integers(0, K, N)
    B = np.zeros((K, N))
    B[pick, np.arange(N)] = 1.0
    got = _call(ttsn, A.T.copy() if ta else A, B.T.copy() if tb else B, ta, tb)
    assert np.array_equal(got, A[:, pick])


@pytest.mark.parametrize("m,n", [(900, 140), (30001, 65)])
def test_gram_of_columns_that_are_large_at_different_rows(ttsn, m, n):
    """Positive entries: the FP64 pipe's sums are off by m eps relative at most,
    and so is the reference's."""
    import torch

    rng = np.random.default_rng(m)
    A = 1e-18 * (1.0 + rng.random((m, n)))
    A[np.arange(n) * (m // n), np.arange(n)] = 1.0
    G = ttsn.gram(torch.as_tensor(A, device="cuda")).cpu().numpy()
    ref = A.T @ A
    assert np.all(np.abs(G - ref) <= 2 * m * np.finfo(float).eps * ref) and np.array_equal(G, G.T)


@pytest.mark.parametrize("r1,r2", [(46, 20), (52, 48), (64, 24)])
def test_captured_steps_that_split_where_their_capacity_does_not(ttsn, r1, r2):
    """256^2 cells, 32 x 64 ordinates, cap 128: the core update and Theta* G_B are
    split at these ranks but not at the cap's sizes.  A short time step keeps the ranks."""
    import torch

    import workloads

    p = workloads.problem("small_2d", n=(256, 256), n_theta=32, n_phi=64, eps=1e-4, bc=1)
    p["max_rank"], p["dt"] = 128, 1e-9
    g = torch.Generator(device="cuda").manual_seed(r1)

    def rnd(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

    # an isotropic field in equilibrium and modes without angular mean, every
    # direction of both bonds well above eps
    X, Th, Ph = 0.05 * rnd(1, 256 * 256, r1), rnd(r1, 32, r2), rnd(r2, 64, 1)
    X[0, :, 0] = torch.as_tensor(p["T0"].reshape(-1), device="cuda") ** 4 / (4 * np.pi)
    Ph -= Ph.mean(1, keepdim=True)
    Ph[0] = 1.0
    Th[0], Th[:, :, 0], Th[0, :, 0] = 0.0, 0.0, 1.0
    a, b = ttsn.TTSN.from_problem(p), ttsn.TTSN.from_problem(p)
    b.set_graph(True)
    for h in (a, b):
        h.set_cores([X, Th, Ph])
        h.set_T(p["T0"])
    for _ in range(2):
        ia, ib = a.step(), b.step()
        assert ia["ranks"] == ib["ranks"] and r1 <= ia["ranks"][1] <= r1 + 1
    for x, y in zip(a.cores(), b.cores()):
        assert torch.equal(torch.as_tensor(x), torch.as_tensor(y))
    (Ea, Ta, ta), (Eb, Tb, tb) = a.energy(), b.energy()
    assert torch.equal(Ea, Eb) and torch.equal(Ta, Tb) and ta == tb


@pytest.mark.parametrize("M,N,K", [(300, 260, 260), (60, 50, 9000)])
def test_product_whose_waits_run_out_is_recomputed(ttsn, M, N, K):
    """Every wait of the digit kernel gives up at once and C is written by nothing
    (written whole, or summed from planes that were not): the FP64 pipe's sum
    replaces it, off by K eps sum |a||b| at most, as is the reference's."""
    import torch

    from paper_2503_18056_gb300 import _native

    rng = np.random.default_rng(M)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    a, b = torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda")
    c = torch.full((M, N), -7.0, dtype=torch.float64, device="cuda")
    st = _native.lib.tt_digits_wait_probe(M, N, K, *(ctypes.c_void_p(x.data_ptr()) for x in (a, b, c)),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    assert np.all(np.abs(c.cpu().numpy() - A @ B) <= 2 * K * np.finfo(float).eps * (np.abs(A) @ np.abs(B)))
    assert torch.equal(torch.as_tensor(_call(ttsn, A, B, False, False), device="cuda"), ttsn.dgemm(a, b))


def test_rows_that_cannot_be_split_leave_the_others_as_they_are(ttsn):
    """A row below 2^-900 or with an Inf and a column with a NaN are recomputed with
    their 16 x 16 tiles; every other entry keeps the digit product's bits."""
    rng = np.random.default_rng(1)
    M, N, K = 300, 260, 300
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    plain = _call(ttsn, A, B, False, False)
    X, Y = A.copy(), B.copy()
    X[37] *= 1e-290
    X[120, 5] = np.inf
    Y[9, 201] = np.nan
    got = _call(ttsn, X, Y, False, False)
    with np.errstate(all="ignore"):
        ref = X @ Y
    rows, cols = np.ones(M, bool), np.ones(N, bool)
    rows[32:48] = rows[112:128] = cols[192:208] = False
    assert np.array_equal(got[np.ix_(rows, cols)], plain[np.ix_(rows, cols)])
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    fine = np.isfinite(ref)
    bound = (K + 1) * np.finfo(float).eps * (np.abs(A) @ np.abs(B))
    bound[37] *= 1e-290
    assert np.all(np.abs(got[fine] - ref[fine]) <= 2 * bound[fine])


@pytest.mark.parametrize("rows", [262144, 2097152])
@pytest.mark.parametrize("where", ["one", "patch", "scattered"])
@pytest.mark.parametrize("eps", [1e-6, 1e-7])
def test_rounding_of_point_like_columns_keeps_its_tolerance(ttsn, rows, where, eps):
    """Large entries in a few rows over a background of 2^-28, whose singular values are
    1e-8 to 1e-6 of the norm: one scale a column would lose the background's products.
    The rounding must do as well as with a Gram from FP64 sums (gram_noalloc, with the
    same eigensolver and truncation), which itself cannot resolve all of these."""
    import torch

    n = 40
    r = torch.arange(rows, device="cuda", dtype=torch.float64)
    f = torch.arange(1, n + 1, device="cuda", dtype=torch.float64)
    A = 2.0 ** -28 * torch.cos(2 * np.pi * (r[:, None] + 0.5) * f[None, :] / rows)
    at = {"one": [12345], "patch": range(70000, 70006), "scattered": range(100, rows, rows // 60)}[where]
    A[list(at)] += 1.0
    tt = ttsn.TensorTrain([A[None].contiguous(), torch.eye(n, device="cuda", dtype=torch.float64)[:, :, None].contiguous()])
    tt.round(eps=eps)
    err = float(torch.linalg.norm(tt.full().reshape(rows, n) - A) / torch.linalg.norm(A))
    lam, V, _ = ttsn.syev_psd(ttsn.gram_noalloc(A))
    tail = torch.flip(torch.cumsum(torch.flip(lam, (0,)), 0), (0,))
    r64 = min(int((tail > eps * eps * lam.sum()).sum()), int((lam > n * 2.0 ** -52 * lam[0]).sum()))
    err64 = float(torch.linalg.norm(A - (A @ V[:r64].T) @ V[:r64]) / torch.linalg.norm(A))
    assert err <= 1.1 * max(eps, err64)


def test_gram_of_long_columns_whose_blocks_differ_in_scale(ttsn):
    """Blocks of 512 rows scaled by powers of two, a few of them far below the others,
    integer entries, so every block's sum is an integer times a power of two.  The sum
    is off by its last rounding and, for each of the 80 blocks, by at most 2^-71 of
    2^(e_i + e_j) <= 16 max|a_i| max|a_j|."""
    import torch

    rng = np.random.default_rng(3)
    m, n = 40960, 48
    A = rng.integers(-(1 << 12), 1 << 12, (m, n)).astype(float)
    down = np.where(np.arange(m // 512) % 8 == 3, rng.integers(10, 61, m // 512), rng.integers(0, 5, m // 512))
    s = 2.0 ** -np.repeat(down, 512)[:, None].astype(float)
    G = ttsn.gram(torch.as_tensor(A * s, device="cuda")).cpu().numpy()
    ref = np.zeros((n, n), np.longdouble)
    for b in range(m // 512):
        blk = A[512 * b:512 * b + 512].astype(np.int64)
        ref += (blk.T @ blk).astype(np.longdouble) * np.longdouble(s[512 * b, 0]) ** 2
    mx = np.abs(A * s).max(0)
    assert np.all(np.abs(G - ref) <= 80 * 2.0 ** -67 * mx[:, None] * mx[None, :] + 2.0 ** -53 * np.abs(ref))
    assert np.array_equal(G, G.T)


def _gauged(rng, shape, ranks, decades):
    """Cores of a TT, and those of the same tensor with a graded power-of-two gauge on
    every bond."""
    r = [1] + ranks + [1]
    cores = [rng.standard_normal((r[k], shape[k], r[k + 1])) for k in range(len(shape))]
    other = [c.copy() for c in cores]
    for k in range(len(shape) - 1):
        D = 2.0 ** np.round(decades * np.log2(10.0) * rng.random(r[k + 1]))
        other[k] *= D
        other[k + 1] /= D[:, None, None]
    return cores, other


def test_graded_gauge_does_not_change_the_full_tensor(ttsn):
    """Scaling a core's columns by D and the next core's rows by 1 / D, powers of two
    over eight decades, changes no rounding error of a sum over the bond."""
    import torch

    cores, other = _gauged(np.random.default_rng(7), (3000, 64, 40), [90, 90], 8)
    assert torch.equal(ttsn.TensorTrain(cores).full(), ttsn.TensorTrain(other).full())


def test_rounding_with_a_graded_gauge_gives_an_orthonormal_core(ttsn):
    """A' = A P_A with P_A from the eigenvectors of K = W G_A W^T: its columns are
    orthonormal to the rounding of K, n^2 eps lambda_1, relative to its smallest
    eigenvalue, whatever the bonds' gauge (six decades here); with a scale a row and
    not the bond's, the digit products would lose the gauge's decades."""
    import torch

    cores, other = _gauged(np.random.default_rng(8), (3000, 64, 40), [90, 90], 6)
    for c in (cores, other):
        tt = ttsn.TensorTrain(c)
        X = tt.full().reshape(3000, -1)
        tt.round(eps=1e-6)
        A = tt.cores()[0].reshape(3000, -1)
        r = A.shape[1]
        sv = torch.linalg.svdvals(X)
        bound = 90 ** 2 * 2.0 ** -52 * float(sv[0] / sv[r - 1]) ** 2
        assert r == 90 and bound < 1e-9
        assert float((A.T @ A - torch.eye(r, device=A.device, dtype=A.dtype)).abs().max()) <= bound
        assert float(torch.linalg.norm(tt.full().reshape(3000, -1) - X) / torch.linalg.norm(X)) <= 1e-6


def test_full_tensor_with_an_index_that_one_core_does_not_have(ttsn):
    """A row of zeros in one core against a column that is 2^40 above the other core's
    columns: it adds nothing and must not set the scale of what does.  A term is off by
    9.1 2^-58 2^(e_i + e_j) at most, the exponents those of entries scaled by m_k, the
    largest of core 2's row k (a power of two at most 2 away, twice): under 2^-48 max_k(|a_ik|
    m_k) max_k(|b_kj| / m_k)."""
    rng = np.random.default_rng(11)
    K = 90
    A, B = 2.0 ** -40 * rng.standard_normal((3000, K)), rng.standard_normal((K, 2560))
    A[:, 0], B[0] = rng.standard_normal(3000), 0.0
    got = ttsn.TensorTrain([A[None], B[:, :, None]]).full().reshape(3000, 2560).cpu().numpy()
    m = np.abs(B[1:]).max(1)
    bound = K * 2.0 ** -48 * (np.abs(A[:, 1:]) * m).max(1)[:, None] * (np.abs(B[1:]) / m[:, None]).max(0)[None, :] \
        + (K + 1) * np.finfo(float).eps * (np.abs(A) @ np.abs(B))
    assert np.all(np.abs(got - A @ B) <= bound)


def test_rounding_with_a_zero_column_gives_an_orthonormal_core(ttsn):
    """A column of zeros (the emission column of a field without absorption) beside
    columns of 2^-40: bounds as with the graded gauge."""
    import torch

    cores, _ = _gauged(np.random.default_rng(12), (3000, 64, 40), [90, 90], 0)
    cores[0] *= 2.0 ** -40
    cores[0][:, :, 0] = 0.0
    tt = ttsn.TensorTrain(cores)
    X = tt.full().reshape(3000, -1)
    tt.round(eps=1e-6)
    A = tt.cores()[0].reshape(3000, -1)
    r = A.shape[1]
    sv = torch.linalg.svdvals(X)
    bound = 90 ** 2 * 2.0 ** -52 * float(sv[0] / sv[r - 1]) ** 2
    assert r == 89 and bound < 1e-9
    assert float((A.T @ A - torch.eye(r, device=A.device, dtype=A.dtype)).abs().max()) <= bound
    assert float(torch.linalg.norm(tt.full().reshape(3000, -1) - X) / torch.linalg.norm(X)) <= 1e-6


@pytest.mark.parametrize("M,K,N", [(3000, 90, 2560), (2560, 300, 300), (300, 2000, 300)])
@pytest.mark.parametrize("which", [0, 1])
def test_full_tensor_of_blocks_at_different_scales(ttsn, M, K, N, which):
    """One core dense, the other of four blocks on their own indices, nine decades
    apart: no scale of the index shows the small blocks' products to the dense core's
    rows, so those are recomputed.  What is not has K / 18 indices at least where both
    entries are within 2^-9 of the exponents, where a term is off by 9.1 2^-58: under
    2^-30 of the sum |a||b|."""
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    X = A if which else B
    m, n = X.shape
    keep = np.zeros((m, n))
    for i in range(4):
        keep[i * m // 4:(i + 1) * m // 4, i * n // 4:(i + 1) * n // 4] = 10.0 ** (-3 * i)
    X *= keep
    got = ttsn.TensorTrain([A[None], B[:, :, None]]).full().reshape(M, N).cpu().numpy()
    assert np.all(np.abs(got - A @ B) <= (2.0 ** -30 + (K + 1) * np.finfo(float).eps) * (np.abs(A) @ np.abs(B)))
