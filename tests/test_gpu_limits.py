"""Limits of buffers and launches: the longest rows that the slicers take through shared memory,
exchange partials of a basis with few occupied orbitals, the workspace cap, the choice of tile
widths set and read back, the rounding of the one-electron energy, and results whose rows are far
apart."""
import numpy as np
import pytest

from gpu_common import built, dev, gpu_energy_grad, make_las, torch_cuda
from las_inputs import make_system
from oracle import las_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch_cuda()
    built()


# The row buffer of the K-major slicers ends at 383 K blocks (6128 values); with their static shared
# memory of 1 and 2 KB that is more than the 48 KB a kernel has without asking for more, from 368 and
# 376 blocks on (5873 and 6001 values).
@pytest.mark.parametrize("K", [5856, 5872, 5873, 5984, 6000, 6001, 6064, 6065, 6112, 6113, 6128, 6129])
def test_split_gemm_longest_rows_in_shared_memory(K):
    from paper_2505_03755_gb300 import split_gemm
    rng = np.random.default_rng(K)
    for M in (1, 40):
        A, B = rng.standard_normal((M, K)), rng.standard_normal((K, 30))
        # operand rounding, dropped digit pairs and FP32 tails: below 2^-43 K rowmax colmax
        bound = 2.0 ** -43 * K * np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :]
        C = split_gemm(dev(A), dev(B)).cpu().numpy()
        assert np.all(np.abs(C - A @ B) <= bound)


# (auxiliary rows) x (padded occupied columns) of a chunk is the length of the projection's W rows:
# 5984 to 6144 in steps of 16, and two lengths at the widest tile and at several tiles
@pytest.mark.parametrize("n,c,X", [(20, 4, X) for X in range(374, 385)] +
                         [(100, 88, 63), (150, 139, 42)])
def test_energy_grad_longest_projection_rows(n, c, X):
    s = make_system(n, X, c, [(2, 2), (2, 3)], seed=X)
    ref = O.system_energy_grad(s)
    for precision in ("split", "split_packed"):
        E, G, g = gpu_energy_grad(s, precision)
        assert abs(E - ref["E"]) <= 1e-8
        assert np.abs(G - ref["G"]).max() <= 1e-8
        assert np.abs(g - ref["gorb"]).max() <= 1e-7


# More than 64 basis functions per padded occupied column: one n x n partial of the exchange is larger
# than the projection's partials.  1030 orbitals also leave 6 rows past the last row tile, and 1024
# (no more than 64 per column) is the other side of the edge.
@pytest.mark.parametrize("n", [1024, 1030, 1152])
@pytest.mark.parametrize("precision", ["split", "split_packed"])
def test_exchange_with_few_occupied_orbitals(n, precision):
    s = make_system(n, 5, 8, [(2, 2), (2, 3)], seed=n)
    las = make_las(s, precision)
    (Jr,), (Kr,) = O.df_jk(s.Bp, n, [2.0 * s.C[:, :8] @ s.C[:, :8].T])
    J, K = las.df_jk(dev(s.C))
    las.sync()
    assert np.abs(J.cpu().numpy() - Jr).max() <= 1e-11 * np.abs(Jr).max()
    assert np.abs(K.cpu().numpy() - Kr).max() <= 1e-11 * np.abs(Kr).max()
    # densities of both spins, one with a weight of the other sign
    Cx, w = np.ascontiguousarray(s.C[:, :13]), np.linspace(1.0, 0.4, 13)
    wb = np.where(np.arange(13) < 9, w, -w)
    va_r, vb_r = O.embedding_potentials(s.Bp, n, Cx * w @ Cx.T, Cx * wb @ Cx.T)
    va, vb = las.veff(dev(Cx), dev(w), dev(Cx), dev(wb))
    las.sync()
    for v, ref in ((va, va_r), (vb, vb_r)):
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    las.close()


# n = 200, X = 1600, one fragment of 24 orbitals: the partial sums of the Coulomb matrix and the
# transposed 2-RDM are each larger than what the plan leaves unused of the K-split partials
@pytest.mark.parametrize("rows", [1600, 800, 200, 25])
def test_workspace_cap_holds_every_buffer(rows):
    torch = torch_cuda()
    from paper_2505_03755_gb300 import LasDF
    n, X, c, m, op = 200, 1600, 4, 24, 32
    npair, ndm1, ndm2 = n * (n + 1) // 2, 2 * m * m, m ** 4
    g = torch.Generator(device="cuda")
    g.manual_seed(rows)
    B = torch.randn(X, npair, generator=g, device="cuda", dtype=torch.float64)
    C = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    # what the plan counts, with the chunk of `rows` auxiliary rows that it then chooses
    cap = 8 * (4 * n * op + 256 + n * op + 3 * X + npair + ndm2 + 64 * n * op
               + rows * op * (n + 2 * op))
    out = []
    for limit in (0, cap):
        las = LasDF(B, n, X, n, c, [m], precision="fp64", max_workspace_bytes=limit)
        # beside the workspace: the staging buffers of the host-buffer call
        staging = 8 * (2 * n * n + n * n + ndm1 + ndm2)
        if limit:
            assert las.device_bytes() - staging <= limit
        J, K = las.df_jk(C)
        las.sync()
        out.append((J.cpu().numpy(), K.cpu().numpy()))
        las.close()
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()


@pytest.mark.parametrize("precision", ["split", "split_packed"])
def test_tile_widths_round_trip(precision):
    """What tiles() returns can be set again and restores the same choice: 0 stands for the library's
    rule, in force until a width is set."""
    s = make_system(60, 80, 30, [(2, 2), (2, 3)], seed=60)
    las = make_las(s, precision)
    args = (dev(s.C), dev(s.h), dev(s.dm1s_flat()), dev(s.dm2_flat()))

    def evaluate():
        E, G = las.energy_grad(*args)
        las.sync()
        return float(E), G.cpu().numpy()

    first = las.tiles()
    assert first == [0, 0, 0, 0]
    e0, g0 = evaluate()
    for widths in ([96, 64, 96, 64], [0, 96, 0, 64], first):
        las.set_tiles(widths)
        assert las.tiles() == widths
        e, g = evaluate()
        assert e == e0 and np.array_equal(g, g0)
    las.autotune(*args)
    chosen = las.tiles()
    las.set_tiles(chosen)
    assert las.tiles() == chosen
    for bad in (48, 80, -64, 1):
        with pytest.raises(Exception):
            las.set_tiles([bad, 96, 96, 96])
    assert las.tiles() == chosen
    las.close()


def test_one_electron_energy_is_compensated():
    """Row 0 holds 2^60, 1 and -2^60 in columns 0, 32 and 64, and row 1 again: a sum that does not
    carry its rounding errors loses the ones.  All values and their products are exact; E = 4."""
    from paper_2505_03755_gb300 import LasDF
    n, c, X = 70, 67, 2
    B, h, C = np.zeros((X, n * (n + 1) // 2)), np.zeros((n, n)), np.zeros((n, n))
    h[0, 1] = h[1, 0] = 2.0 ** 60
    C[0, [0, 32, 64]] = 1.0
    C[1, [0, 32, 64]] = 1.0, 2.0 ** -60, -1.0
    las = LasDF(dev(B), n, X, n, c, [], precision="fp64")
    E = las.energy(dev(C), dev(h), dev(np.zeros(0)), dev(np.zeros(0)))
    las.sync()
    assert float(E) == 4.0
    las.close()


@pytest.mark.parametrize("K", [1041, 40])
def test_split_gemm_rows_of_the_result_far_apart(K):
    """A leading dimension of C beyond 2^31 values (a product that is split over K, and one that is
    not): the two rows land where they belong."""
    torch = torch_cuda()
    from paper_2505_03755_gb300 import load_library
    lib = load_library()
    M, N, ldc = 2, 5, 2 ** 31 + 8
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 18 GB")
    rng = np.random.default_rng(K)
    A, B = np.rint(50 * rng.standard_normal((M, K))), np.rint(50 * rng.standard_normal((K, N)))
    a, b = dev(A), dev(B)
    c = torch.empty((M - 1) * ldc + N, dtype=torch.float64, device="cuda")
    need = lib.las_split_gemm_workspace(M, N, K)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert lib.las_split_gemm(M, N, K, a.data_ptr(), K, b.data_ptr(), N, c.data_ptr(), ldc,
                              ws.data_ptr(), need, st) == 0
    got = torch.stack([c[:N], c[ldc:ldc + N]]).cpu().numpy()
    del c
    torch.cuda.empty_cache()
    assert np.array_equal(got, A @ B)
