"""FP64 products and block inverses on the tensor cores (nine digit planes) against extended precision.

Bar of a product: each operand value is held to 2^-62 of its row's or column's largest entry (2^-61 for
K > 256), digit products beyond i + j = 10 are dropped (below 2^-56 of the leading digits' product), and
the sum is rounded to FP64 once: |C - C_exact| <= 2^-53 |C| + K 2^-54 max|A_row| max|B_col| covers it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2606_25595_gb300 import build
    build.build()
    import paper_2606_25595_gb300 as q
    q.load()
    return q


def _cx(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _ld(x):
    return x.astype(np.clongdouble)


# edges of the tiles (33, 128, 129 rows; 32-column tiles and their 8-column remainder), of the K padding
# and of one launch's contraction (512, then chunks)
@pytest.mark.parametrize("M,N,K", [(33, 33, 33), (48, 40, 47), (64, 65, 64), (128, 32 * 5, 256), (129, 97, 257),
                                   (200, 121, 130), (60, 250, 512), (40, 40, 513), (70, 50, 1100)])
@pytest.mark.parametrize("ops", ["NN", "NC", "CN", "CC"])
def test_fp64_product(q, M, N, K, ops):
    import torch
    rng = np.random.default_rng(M * 7 + N + K)
    A = _cx(rng, 2, *((M, K) if ops[0] == "N" else (K, M)))
    B = _cx(rng, 2, *((K, N) if ops[1] == "N" else (N, K))) * 2.0 ** rng.integers(-3, 4)
    C0 = _cx(rng, 2, M, N)
    C = q.zgemm_batched(torch.tensor(A).cuda(), torch.tensor(B).cuda(), "fp64", ops[0], ops[1], alpha=-0.75, beta=0.5,
                        C0=torch.tensor(C0).cuda()).cpu().numpy()
    H = lambda x: np.conj(np.swapaxes(x, 1, 2))  # noqa: E731
    a, b = _ld(A if ops[0] == "N" else H(A)), _ld(B if ops[1] == "N" else H(B))
    ref = -0.75 * np.stack([a[e] @ b[e] for e in range(2)]) + 0.5 * _ld(C0)
    bound = 2.0 ** -52 * (np.abs(ref) + np.abs(C0) * 2) + K * 2.0 ** -54 * np.abs(a).max(2)[:, :, None] * np.abs(b).max(1)[:, None, :]
    assert np.all(np.abs(C - ref) <= bound), float((np.abs(C - ref) / bound).max())


def test_fp64_product_scales_and_specials(q):
    import torch
    rng = np.random.default_rng(5)
    n = 64
    A, B = _cx(rng, 1, n, n), _cx(rng, 1, n, n)
    A[0, 3] *= 1e-200
    A[0, 4] = 0
    B[0, :, 7] *= 1e150
    A[0, 5, 9] = np.inf
    B[0, 2, 11] = np.nan
    C = q.zgemm_batched(torch.tensor(A).cuda(), torch.tensor(B).cuda(), "fp64").cpu().numpy()[0]
    fin = np.ones((n, n), bool)
    fin[5], fin[:, 11] = False, False
    a, b = np.where(np.isfinite(A[0]), A[0], 0), np.where(np.isfinite(B[0]), B[0], 0)
    ref = (_ld(a) @ _ld(b))
    bound = 2.0 ** -52 * np.abs(ref) + n * 2.0 ** -54 * np.abs(a).max(1)[:, None] * np.abs(b).max(0)[None, :]
    assert np.all(np.abs(C - ref)[fin] <= bound[fin])
    assert not np.isfinite(C[5]).any() and np.isnan(C[:, 11]).all() and (C[4][np.isfinite(C[4])] == 0).all()


# values of mixed size inside rows and columns: graded over `decades`, in an order of k shared by A and B (large meets
# large) or opposite (large meets small), and with large values meeting zeros
@pytest.mark.parametrize("K", [64, 300])
@pytest.mark.parametrize("decades", [8, 16, 30])
@pytest.mark.parametrize("meet", ["large", "small", "zeros"])
def test_fp64_product_of_mixed_sizes_within_the_stated_bound(q, K, decades, meet):
    import torch
    rng = np.random.default_rng(K + decades)
    n = 40
    grade = 10.0 ** -np.linspace(0, decades, K)
    A, B = _cx(rng, 1, n, K) * grade, _cx(rng, 1, K, n) * (grade[::-1] if meet == "small" else grade)[:, None]
    if meet == "zeros":
        B[0, : K // 2] = 0
    C = q.zgemm_batched(torch.tensor(A).cuda(), torch.tensor(B).cuda(), "fp64").cpu().numpy()[0]
    ref = _ld(A[0]) @ _ld(B[0])
    bound = 2.0 ** -53 * np.abs(ref) + K * 2.0 ** -54 * np.abs(A[0]).max(1)[:, None] * np.abs(B[0]).max(0)[None, :]
    assert np.all(np.abs(C - ref) <= bound), float((np.abs(C - ref) / bound).max())


def test_fp64_product_error_not_above_dfma(q):
    """Error against exact rational sums, beside that of a plain FP64 product (the library's own below
    33 rows is DFMA: the same operands, 32 rows at a time)."""
    import torch
    from fractions import Fraction
    rng = np.random.default_rng(6)
    for n in (48, 128, 256):
        A, B = _cx(rng, 1, n, n), _cx(rng, 1, n, n)
        tA, tB = torch.tensor(A).cuda(), torch.tensor(B).cuda()
        C = q.zgemm_batched(tA, tB, "fp64").cpu().numpy()[0]
        D = q.zgemm_batched(tA[:, :32].contiguous(), tB, "fp64").cpu().numpy()[0]
        ec = ed = 0.0
        for i in range(2):
            for j in range(0, n, 4):
                x = sum(Fraction(a.real) * Fraction(b.real) - Fraction(a.imag) * Fraction(b.imag)
                        for a, b in zip(A[0, i], B[0, :, j]))
                ec += float(Fraction(C[i, j].real) - x) ** 2
                ed += float(Fraction(D[i, j].real) - x) ** 2
        assert ec <= ed, (n, ec, ed)


@pytest.mark.parametrize("prec", ["fp64", "emu64"])
def test_product_strides_and_overlap(q, prec):
    """Padded rows and gapped batches; C0 = C; C on top of an operand still gives the product (emulated
    FP64: to its 2^-36 of the operands' magnitudes)."""
    import ctypes
    import torch
    rng = np.random.default_rng(8)
    M, N, K, bt = 50, 40, 60, 3
    A, B = torch.tensor(_cx(rng, bt + 1, M, K + 5)).cuda(), torch.tensor(_cx(rng, 1, N, K + 3)).cuda()
    C = torch.tensor(_cx(rng, bt, M, N + 2)).cuda()
    C0 = C.clone()
    L = q.load()
    p, atol = q.PRECISION[prec], 1e-13 if prec == "fp64" else 1e-8
    st = L.qtx_zgemm_batched(p, M, N, K, 0, A.data_ptr(), K + 5, M * (K + 5), 1, B.data_ptr(), K + 3, 0, 1.0, 1.0,
                             C.data_ptr(), N + 2, M * (N + 2), C.data_ptr(), N + 2, M * (N + 2), bt,
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    ref = C0.clone()
    ref[:, :, :N] += A[:bt, :, :K] @ B[0, :, :K].conj().T
    assert torch.allclose(C, ref, rtol=1e-14, atol=atol)
    X, Y = torch.tensor(_cx(rng, 2, 64, 64)).cuda(), torch.tensor(_cx(rng, 2, 64, 64)).cuda()
    ref = X @ Y
    st = L.qtx_zgemm_batched(p, 64, 64, 64, 0, X.data_ptr(), 64, 4096, 0, Y.data_ptr(), 64, 4096, 1.0, 0.0, None, 64, 0,
                             X.data_ptr(), 64, 4096, 2, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0 and torch.allclose(X, ref, rtol=1e-14, atol=atol)


# refined from an FP32 start (33, 64, 200), beyond its reach (kappa 1e9: elimination), a block whose
# leading entries vanish (pivoting), n above the one-CTA elimination
@pytest.mark.parametrize("n,kappa", [(33, 1e2), (64, 1e5), (200, 1e3), (100, 1e9), (257, 1e8)])
def test_fp64_inverse(q, n, kappa):
    import torch
    rng = np.random.default_rng(n)
    U, _ = np.linalg.qr(_cx(rng, n, n))
    V, _ = np.linalg.qr(_cx(rng, n, n))
    A = np.stack([(U * np.geomspace(1, 1 / kappa, n)) @ V, np.eye(n) * (2 - 1j) + _cx(rng, n, n) / n])
    X, st = q.zinv_batched(torch.tensor(A).cuda(), "fp64")
    X = X.cpu().numpy()
    assert (st.cpu().numpy() == 0).all()
    for e in range(2):
        k = np.linalg.cond(A[e])
        ref = np.linalg.inv(A[e])
        assert np.linalg.norm(X[e] - ref) / np.linalg.norm(ref) < 64 * k * 2.0 ** -53


def test_fp64_inverse_pivots_and_singular(q):
    import torch
    n = 40
    rng = np.random.default_rng(1)
    A = np.stack([np.eye(n)[rng.permutation(n)] + 0j, np.zeros((n, n)) + 0j, np.eye(n) * (1 + 1j), np.eye(n) * 1e250 + 0j])
    A[2, 0, 0] = np.nan
    X, st = q.zinv_batched(torch.tensor(A).cuda(), "fp64")
    assert st.cpu().tolist() == [0, 4, 4, 0]
    assert np.array_equal(X[0].cpu().numpy(), A[0].T)
    assert np.allclose(X[3].cpu().numpy() * 1e250, np.eye(n), atol=1e-15)


# beyond FP32's reach (kappa 1e9): eliminated over a cluster's CTAs, whose column ranges and rows do not divide evenly;
# blocks that do (kappa 10), a permutation and a singular block beside them
@pytest.mark.parametrize("n", [33, 64, 65, 131, 255, 256])
def test_fp64_elimination_of_ill_conditioned_blocks(q, n):
    import torch
    rng = np.random.default_rng(n)

    def block(kappa):
        U, _ = np.linalg.qr(_cx(rng, n, n))
        V, _ = np.linalg.qr(_cx(rng, n, n))
        return (U * np.geomspace(1, 1 / kappa, n)) @ V

    P = np.eye(n)[rng.permutation(n)] * (1 + 2j)
    A = np.stack([block(1e9), block(1e9) * 1e-30, P, block(1e1), np.ones((n, n)) + 0j, block(1e9)])
    X, st = q.zinv_batched(torch.tensor(A).cuda(), "fp64")
    X = X.cpu().numpy()
    assert st.cpu().tolist() == [0, 0, 0, 0, 4, 0]
    for e in (0, 1, 2, 3, 5):
        ref = np.linalg.inv(A[e])
        assert np.linalg.norm(X[e] - ref) <= 64 * np.linalg.cond(A[e]) * 2.0 ** -53 * np.linalg.norm(ref), e
    alone, _ = q.zinv_batched(torch.tensor(A[5:]).cuda(), "fp64")
    assert np.array_equal(alone[0].cpu().numpy(), X[5])
