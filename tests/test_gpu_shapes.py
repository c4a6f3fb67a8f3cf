"""Edges of the kernels' tiles and of the rules that choose between them: column widths of the split
product (48 to 96), its K split, rows that start between two 512-byte box rows, rows too long for
shared memory, unaligned rows and results; the FP64 GEMM's 16 x 8 blocks; the per-aux kernel's
fragment structures; the exchange product's two forms; the Hessian-vector product without Dg."""
import ctypes

import numpy as np
import pytest

from gpu_common import built, dev, gpu_energy_grad, make_las, torch_cuda
from las_inputs import LasSystem, make_system
from oracle import las_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch_cuda()
    built()


def _bound(A, B):
    # operand rounding 2 x 2^-48, dropped digit pairs 5 x 2^-48 and the FP32 tails 11 x 2^-56 per
    # product term, relative to row and column maxima: below 2^-43 K rowmax colmax
    return 2.0 ** -43 * A.shape[1] * np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :]


# one and several tiles of every width, a column less and a column more; results whose rows are and
# are not 32-byte aligned; one K block, a ragged one, one chunk of 256 and more, and a K that is split
@pytest.mark.parametrize("K", [1, 17, 256, 1041])
@pytest.mark.parametrize("N", [1, 47, 48, 49, 64, 65, 80, 81, 96, 97, 128, 160, 193])
def test_split_gemm_widths(N, K):
    from paper_2505_03755_gb300 import split_gemm
    rng = np.random.default_rng(1000 * N + K)
    for M in (1, 129, 300):
        A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
        C = split_gemm(dev(A), dev(B)).cpu().numpy()
        assert np.all(np.abs(C - A @ B) <= _bound(A, B)), (M, N, K)
        Ai, Bi = np.rint(50 * A), np.rint(50 * B)
        assert np.array_equal(split_gemm(dev(Ai), dev(Bi)).cpu().numpy(), Ai @ Bi), (M, N, K)


# numbers of K blocks around the ends of a chunk's first turn and of a chunk (1, 4, 5, 6, 8, 15, 16, 17,
# 20, 21, 33 blocks of 16), with up to three tiles in a row on one SM
@pytest.mark.parametrize("kb", [1, 4, 5, 6, 8, 15, 16, 17, 20, 21, 33])
@pytest.mark.parametrize("N", [48, 64, 128])
def test_split_gemm_issuer_turns(N, kb):
    from paper_2505_03755_gb300 import split_gemm
    K = 16 * kb - 3
    rng = np.random.default_rng(100 * N + kb)
    A, B = rng.standard_normal((40000, K)), rng.standard_normal((K, N))
    C = split_gemm(dev(A), dev(B)).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= _bound(A, B))
    Ai, Bi = np.rint(50 * A[:20000]), np.rint(50 * B)
    assert np.array_equal(split_gemm(dev(Ai), dev(Bi)).cpu().numpy(), Ai @ Bi)


# the longest row that fits a block's shared memory, one value more (the warp-per-row slicer), and
# rows of odd length (8-byte loads); zero rows; rows of very different scale
@pytest.mark.parametrize("K", [6127, 6128, 6129, 7001])
def test_split_gemm_long_rows(K):
    from paper_2505_03755_gb300 import split_gemm
    rng = np.random.default_rng(K)
    A = rng.standard_normal((40, K)) * 10.0 ** rng.integers(-9, 9, size=(40, 1))
    A[7] = 0.0
    B = rng.standard_normal((K, 30))
    C = split_gemm(dev(A), dev(B)).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= _bound(A, B))
    assert np.all(C[7] == 0.0)


def test_split_gemm_workspace_without_partials():
    """A workspace that holds the digit planes only (the least that was ever asked for) still
    serves: the K split then goes without its partials."""
    torch = torch_cuda()
    from paper_2505_03755_gb300 import load_library, split_gemm
    lib = load_library()
    M, N, K = 300, 70, 1041
    rng = np.random.default_rng(5)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    rup = lambda x, m: (x + m - 1) // m * m
    planes = lambda R: rup(6 * rup(R, 384) * ((K + 15) // 16) * 16 * 2, 256)
    least = planes(M) + planes(N) + rup(4 * M, 256) + rup(4 * N, 256) + 256
    assert lib.las_split_gemm_workspace(M, N, K) > least      # this product is split
    a, b = dev(A), dev(B)
    c = torch.empty((M, N), dtype=torch.float64, device="cuda")
    ws = torch.empty(least, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    for nbytes, want in ((least, 0), (least - 256, 3)):
        assert lib.las_split_gemm(M, N, K, a.data_ptr(), K, b.data_ptr(), N, c.data_ptr(), N,
                                  ws.data_ptr(), nbytes, st) == want
    assert np.all(np.abs(c.cpu().numpy() - A @ B) <= _bound(A, B))
    assert np.all(np.abs(split_gemm(a, b).cpu().numpy() - A @ B) <= _bound(A, B))


# occupied columns (and the half transform's N) around the FP64 GEMM's 8-column blocks and its widest
# tile, orbitals around its 16-row blocks and 64-row tiles; the split modes over the same shapes,
# with chunks of auxiliary rows that start between two box rows
@pytest.mark.parametrize("n,c,frags", [(15, 3, [(2, 2)]), (16, 0, [(2, 3)]), (33, 7, []),
                                       (64, 37, [(2, 3)]), (65, 38, [(2, 3)]), (97, 79, [(2, 2)]),
                                       (130, 90, [(4, 4), (2, 3)])])
def test_shapes_all_precisions(n, c, frags):
    s = make_system(n, 45, c, frags, seed=n)
    ref = O.system_energy_grad(s)
    for precision, e_tol, g_tol in (("fp64", 1e-10 * abs(ref["E"]), 1e-9), ("split", 1e-8, 1e-8),
                                    ("split_packed", 1e-8, 1e-8)):
        E, G, g = gpu_energy_grad(s, precision)
        assert abs(E - ref["E"]) <= e_tol
        assert np.abs(G - ref["G"]).max() <= g_tol
        assert np.abs(g - ref["gorb"]).max() <= 10 * g_tol
        if precision != "fp64":
            # chunks of about 12 auxiliary rows: products that start at rows such as 12 n, 24 n
            las = make_las(s, precision, max_workspace_bytes=_cap(s, 12))
            G2 = las.energy_grad(dev(s.C), dev(s.h), dev(s.dm1s_flat()), dev(s.dm2_flat()))[1]
            las.sync()
            assert np.abs(G2.cpu().numpy() - ref["G"]).max() <= g_tol
            las.close()


def _cap(s, rows):
    """A workspace cap under which about `rows` auxiliary rows make a chunk (the plan halves the
    chunk until fixed parts, partials and the chunk fit)."""
    n, op = s.nao, (s.nocc + 15) // 16 * 16
    per = 8 * op * (n + 2 * op) + 24 * op * ((n + 15) // 16 * 16) + 12 * 384 * op + 4 * op
    fixed = 8 * (4 * n * op + op * op + s.nmo * op + 3 * s.naux + n * (n + 1) // 2 + 256)
    return fixed + 64 * n * op * 8 + rows * per


def _random_state(n, X, c, ms, seed):
    """A system with arbitrary symmetric RDM blocks (the contractions are linear in them), for
    fragments too large to expand in determinants."""
    s = make_system(n, X, c, [], seed=seed)
    rng = np.random.default_rng(seed)
    s = LasSystem(**{**s.__dict__, "nact": list(ms), "nelec": [0] * len(ms)})
    for m in ms:
        g = rng.standard_normal((2, m, m)) / m
        s.dm1s.append(g + g.transpose(0, 2, 1))
        G = rng.standard_normal((m * m, m * m)) / m ** 2
        G = (G + G.T).reshape(m, m, m, m)
        s.dm2.append(G + G.transpose(1, 0, 3, 2))
    return s


# one-orbital fragments, many fragments, one fragment of all, and two fragments whose blocks leave
# no room in shared memory for the factored cross-fragment path (the direct form)
@pytest.mark.parametrize("ms", [[1], [1, 1, 1], [1, 5, 2, 7, 1], [2] * 20, [33], [60, 30]])
def test_fragment_structures(ms):
    n = max(30, sum(ms) + 6)
    s = _random_state(n, 6, 4, ms, seed=sum(ms))
    ref = O.system_energy_grad(s)
    scale = max(1.0, np.abs(ref["G"]).max())
    for precision, tol in (("fp64", 1e-12), ("split", 1e-10)):
        E, G, _ = gpu_energy_grad(s, precision)
        assert abs(E - ref["E"]) <= tol * max(1.0, abs(ref["E"]))
        assert np.abs(G - ref["G"]).max() <= tol * scale


@pytest.mark.parametrize("n,X,c", [(136, 60, 16), (272, 40, 20), (784, 120, 64)])
@pytest.mark.parametrize("precision", ["split", "split_packed"])
def test_exchange_few_rows_past_a_tile(n, X, c, precision):
    """n = 128 k + 8 or 16: the last rows alone would make a row tile of padding.  At 784 orbitals
    and 7680 rows (L, k) they run as the columns of a second product; at the smaller sizes one
    product ends sooner."""
    s = make_system(n, X, c, [(2, 2)], seed=n)
    D = 2.0 * s.C[:, :c] @ s.C[:, :c].T
    (Jr,), (Kr,) = O.df_jk(s.Bp, n, [D])
    las = make_las(s, precision)
    J, K = las.df_jk(dev(s.C))
    las.sync()
    J, K = J.cpu().numpy(), K.cpu().numpy()
    las.close()
    assert np.abs(J - Jr).max() <= 1e-11 * np.abs(Jr).max()
    assert np.abs(K - Kr).max() <= 1e-11 * np.abs(Kr).max()
    assert np.array_equal(K, K.T) and np.array_equal(J, J.T)


@pytest.mark.parametrize("precision", ["fp64", "split", "split_packed"])
def test_hvp_without_rotation_gradient(precision):
    """dG does not depend on whether Dg (and with it G) is formed, with one chunk and several."""
    s = make_system(37, 53, 5, [(2, 3), (3, 2)], seed=77)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((37, 37))
    X = dev((X - X.T) / np.linalg.norm(X))
    args = (dev(s.C), dev(s.h), dev(s.dm1s_flat()), dev(s.dm2_flat()), X)
    out = []
    for cap in (0, _cap(s, 12)):
        las = make_las(s, precision, max_workspace_bytes=cap)
        a, Dg = las.orbital_hvp(*args)
        b, none = las.orbital_hvp(*args, want_Dg=False)
        las.sync()
        assert none is None and torch_cuda().equal(a, b)
        out.append((a.cpu().numpy(), Dg.cpu().numpy()))
        las.close()
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 1e-9 * np.abs(x).max()


@pytest.mark.parametrize("precision", ["fp64", "split", "split_packed"])
def test_auxiliary_rows_of_extreme_scale(precision):
    """Auxiliary rows of 2^-560 (their products underflow), 2^-1010 (some elements subnormal) and zeros
    beside ordinary ones: the scaling of W by powers of two ends in zero there, with no wrap of the
    exponent field."""
    s = make_system(37, 12, 5, [(2, 3), (3, 2)], seed=78)
    Bp = s.Bp.reshape(12, -1).copy()
    Bp[3] *= 2.0 ** -560
    Bp[5] *= 2.0 ** -1010
    Bp[7] = 0.0
    s.Bp = Bp.reshape(s.Bp.shape)
    ref = O.system_energy_grad(s)
    E, G, _ = gpu_energy_grad(s, precision)
    assert abs(E - ref["E"]) <= (1e-10 * abs(ref["E"]) if precision == "fp64" else 1e-8)
    assert np.abs(G - ref["G"]).max() <= (1e-9 if precision == "fp64" else 1e-8)


def test_fp64_nan_and_infinity_reach_every_result():
    """One NaN or infinity in B makes the energy and every occupied column of dE/dC non-finite: T_L
    has no finite element, and neither has W_L."""
    for bad in (np.nan, np.inf, -np.inf):
        s = make_system(37, 12, 5, [(2, 3), (3, 2)], seed=79)
        Bp = s.Bp.reshape(12, -1).copy()
        Bp[4, 100] = bad
        s.Bp = Bp.reshape(s.Bp.shape)
        E, G, _ = gpu_energy_grad(s, "fp64")
        assert not np.isfinite(E)
        assert not np.isfinite(G[:, :s.nocc]).any()
