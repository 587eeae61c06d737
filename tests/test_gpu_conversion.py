"""Conversion steps (Sec. 4.2, 4.3; App. B, C, D) through the C ABI against the fp64 conversion oracle.

Every step is compared with the oracle's same step on the same inputs.  Eigenvectors are unique only up to sign
(and up to rotation inside a repeated eigenvalue), so they are checked through what is unique: the eigenvalues,
orthonormality, the residual A V - V diag(w), and the energy a leading block captures."""
import numpy as np
import pytest
import torch

from oracle import conversion_oracle as cv
from oracle import mla_oracle as orc
from paper_2502_07864_b200 import binding, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device='cuda')


def _f64(t):
    return t.detach().cpu().numpy().astype(np.float64)


def _rel(got, want):
    return np.linalg.norm(got - want) / max(np.linalg.norm(want), 1e-30)


@pytest.mark.parametrize('ta,tb', [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_gemm_all_storage_orders_with_ragged_edges(ta, tb):
    gu.ensure_built()
    rng = np.random.default_rng(10 + 2 * ta + tb)
    M, N, K = 261, 130, 77
    a = rng.standard_normal((K, M) if ta else (M, K)).astype(np.float32)
    b = rng.standard_normal((N, K) if tb else (K, N)).astype(np.float32)
    c = torch.full((M, N), float('nan'), device='cuda')
    binding.transmla_conv_gemm(_dev(a), _dev(b), c, ta=bool(ta), tb=bool(tb), alpha=0.5)
    want = 0.5 * (a.astype(np.float64).T if ta else a.astype(np.float64)) @ (b.astype(np.float64).T if tb else b.astype(np.float64))
    assert _rel(_f64(c), want) < 1e-6


@pytest.mark.parametrize('M,N,K,ta,tb', [(128, 128, 32, 0, 1), (129, 127, 33, 1, 0), (1, 1, 1, 0, 0), (20000, 301, 100, 0, 1),
                                         (301, 20000, 65, 1, 0), (5001, 5001, 300, 1, 0), (200, 200, 300, 1, 0), (333, 333, 40, 0, 1)])
def test_gemm_tiles_pairs_and_symmetric_products(M, N, K, ta, tb):
    # one tile and one past it; enough tiles for the two-CTA kernel (row strides that are and are not whole 16 bytes); X^T X
    # and X X^T, whose upper half is mirrored.  Per chunk of 32 at most 12 truncations of 2^-23 in the accumulator, then
    # rounded sums: below 1e-6 of the norm for random signs.
    gu.ensure_built()
    gen = torch.Generator(device='cuda'); gen.manual_seed(M + K)
    a = torch.randn((K, M) if ta else (M, K), generator=gen, device='cuda')
    b = a if M == N and ta != tb and M > 129 else torch.randn((N, K) if tb else (K, N), generator=gen, device='cuda')
    c = torch.full((M, N), float('nan'), device='cuda')
    binding.transmla_conv_gemm(a, b, c, ta=bool(ta), tb=bool(tb))
    want = (a.double().T if ta else a.double()) @ (b.double().T if tb else b.double())
    assert float((c - want).norm() / want.norm()) < 1e-6
    if b is a:
        assert torch.equal(c, c.T)


@pytest.mark.parametrize('M,N,K,ta,tb', [(200, 150, 100, 0, 0), (200, 150, 100, 1, 1), (6000, 5000, 40, 0, 1)])
def test_gemm_of_infinities_and_of_values_at_the_ends_of_fp32(M, N, K, ta, tb):
    # one CTA a tile and CTA pairs: values that bf16 terms cannot hold take part as in fp32 arithmetic
    gu.ensure_built()
    gen = torch.Generator(device='cuda'); gen.manual_seed(M)
    a = torch.randn((K, M) if ta else (M, K), generator=gen, device='cuda'); b = torch.randn((N, K) if tb else (K, N), generator=gen, device='cuda')
    op_a, op_b = (a.T if ta else a), (b.T if tb else b)
    c = torch.empty(M, N, device='cuda')

    def run(alpha=1.0):
        binding.transmla_conv_gemm(a, b, c, ta=bool(ta), tb=bool(tb), alpha=alpha)
        return op_a.double() @ op_b.double()

    keep = a.clone()
    op_a[3, 5], op_a[130, 7], op_a[131, 0] = float('inf'), float('-inf'), float('nan')
    op_b[5, 9] = 0.0                                   # inf * 0
    want = run().float()
    assert torch.equal(torch.isnan(c), torch.isnan(want)) and torch.equal(torch.isinf(c), torch.isinf(want))
    assert torch.equal(c.sign()[torch.isinf(c)], want.sign()[torch.isinf(want)])
    ok = torch.isfinite(want)
    assert float((c[ok] - want[ok]).norm() / want[ok].norm()) < 1e-6
    a.copy_(keep); op_a[2], op_b[:, 4] = 3.4e38, 1e-3  # finite, above the largest bf16 value
    want = run(alpha=1e-4)
    got, ref = c[2].double(), want[2] * 1e-4
    fin = torch.isfinite(got)                          # (sums beyond 3.4e38 overflow, as fp32 sums do)
    assert bool(fin[4]) and abs(float(got[4] / ref[4]) - 1) < 1e-5 and float((got[fin] / ref[fin] - 1).abs().max()) < 1e-3
    # small operands: exact terms down to 2^-110, plain sums below; each row's error against its own norm, where a chain of
    # K fp32 multiply-adds keeps K 2^-24 at most
    for scale in (2.0 ** -100, 2.0 ** -112, 2.0 ** -120):
        a.copy_(keep * scale)
        want = run(alpha=2.0 ** 90)
        rel = ((c.double() * 2.0 ** -90 - want).norm(dim=1) / want.norm(dim=1)).max()
        assert float(rel) < K * 2.0 ** -24, scale


@pytest.mark.parametrize('M,N,K,ta,tb,cols', [(200, 150, 100, 0, 0, 32), (200, 150, 100, 1, 1, 32), (6000, 5000, 40, 0, 1, 64),
                                              (5001, 5003, 40, 1, 0, 64)])
@pytest.mark.parametrize('scale', [2.0 ** -112, 2.0 ** -120])
def test_gemm_of_tiny_columns_beside_ordinary_ones(M, N, K, ta, tb, cols, scale):
    # whether tiny operands' sums are taken again is decided for a quarter of a tile's columns (32 of one CTA's, 64 of a
    # pair's): every other quarter tiny, each column's error against its own norm, K 2^-24 at most as a chain of fp32
    # multiply-adds keeps
    gu.ensure_built()
    gen = torch.Generator(device='cuda'); gen.manual_seed(M + cols)
    a = torch.randn((K, M) if ta else (M, K), generator=gen, device='cuda')
    b = torch.randn((N, K) if tb else (K, N), generator=gen, device='cuda')
    op_a, op_b = (a.T if ta else a), (b.T if tb else b)
    tiny = torch.arange(N, device='cuda') // cols % 2 == 0
    op_b[:, tiny] *= scale
    c = torch.empty(M, N, device='cuda')
    binding.transmla_conv_gemm(a, b, c, ta=bool(ta), tb=bool(tb))
    want = op_a.double() @ op_b.double()
    rel = (c.double() - want).norm(dim=0) / want.norm(dim=0)
    assert float(rel.max()) < K * 2.0 ** -24, (float(rel[tiny].max()), float(rel[~tiny].max()))


@pytest.mark.parametrize('pairs,M,N,K', [(0, 100, 90, 500), (0, 300, 1000, 40), (1, 100, 90, 500), (1, 1000, 700, 300)])
def test_gemm_that_gives_up_leaves_no_unfinished_sums(pairs, M, N, K):
    # one CTA a tile and CTA pairs, with waits that expire in every CTA; the launch ends normally
    gu.ensure_built()
    a = torch.randn(M, K, device='cuda'); b = torch.randn(K, N, device='cuda')
    c = torch.zeros(M, N, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    for _ in range(50):
        c.zero_()
        binding.transmla_selftest_conv_gemm(pairs, a, b, c, status)
        assert int(status.item()) & 2                    # TRANSMLA_DEV_TIMEOUT
        assert bool(torch.isnan(c).all())
    binding.transmla_conv_gemm(a, b, c)
    assert _rel(_f64(c), _f64(a) @ _f64(b)) < 1e-6


@pytest.mark.parametrize('ta,tb', [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize('M,N,K', [(1, 1, 1), (129, 260, 1), (300, 131, 4), (128, 128, 16), (130, 257, 17)])
def test_gemm_of_short_sums(M, N, K, ta, tb):
    # up to 16 products a sum: every element within the rounding of K fp32 multiply-adds, K 2^-24 of the sum of sizes
    gu.ensure_built()
    gen = torch.Generator(device='cuda'); gen.manual_seed(M + K)
    a = torch.randn((K, M) if ta else (M, K), generator=gen, device='cuda'); b = torch.randn((N, K) if tb else (K, N), generator=gen, device='cuda')
    c = torch.full((M, N), float('nan'), device='cuda')
    binding.transmla_conv_gemm(a, b, c, ta=bool(ta), tb=bool(tb), alpha=0.5)
    op_a, op_b = (a.T if ta else a).double(), (b.T if tb else b).double()
    # (17 products pass through the split: 12 truncations of 2^-23)
    bound = (K * 2.0 ** -24 if K <= 16 else 12 * 2.0 ** -23) * 0.5 * (op_a.abs() @ op_b.abs())
    assert bool(((c.double() - 0.5 * (op_a @ op_b)).abs() <= bound).all())


@pytest.mark.parametrize('g,d,fold', [(4, 16, 1), (4, 16, 2), (32, 128, 4), (3, 8, 4)])
def test_rorope_covariance_matches_the_oracle(g, d, fold):
    gu.ensure_built()
    rng = np.random.default_rng(20)
    n = 300
    K = rng.standard_normal((n, g * d)).astype(np.float32)
    groups, m = d // 2 // fold, g * fold
    scratch = torch.empty(binding.transmla_conv_rorope_scratch_bytes(n, g, d, fold) // 4, device='cuda')
    cov = torch.full((groups, m, m), float('nan'), device='cuda')
    binding.transmla_conv_rorope_covariance(_dev(K), g, d, fold, scratch, cov)
    want = cv.rorope_covariances(K, g, d, fold)
    assert _rel(_f64(cov), want) < 1e-5


@pytest.mark.parametrize('m,batch', [(7, 3), (32, 64), (128, 4), (1, 2), (2, 1)])
def test_symmetric_eigendecomposition(m, batch):
    gu.ensure_built()
    rng = np.random.default_rng(30 + m)
    x = rng.standard_normal((batch, 3 * m + 2, m)) * (np.arange(1, m + 1) ** -0.7)
    a = np.einsum('bni,bnj->bij', x, x).astype(np.float32)
    w = torch.empty(batch, m, device='cuda'); v = torch.empty(batch, m, m, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    binding.transmla_conv_sym_eig(_dev(a), w, v, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    w, v = _f64(w), _f64(v)
    for b in range(batch):
        want, _ = cv.sorted_eigh(a[b])
        top = want[0]
        assert np.abs(w[b] - want).max() < 2e-5 * top                       # eigenvalues, descending
        assert np.all(np.diff(w[b]) <= 1e-6 * top)
        # orthonormal columns: a column takes part in at most sweeps * (m - 1) fp32 rotations, each off by at most
        # 2^-24 relative; 10 sweeps at m = 128 bound the drift by 8e-5
        assert np.abs(v[b].T @ v[b] - np.eye(m)).max() < 1e-4
        assert np.abs(a[b].astype(np.float64) @ v[b] - v[b] * w[b]).max() < 1e-4 * top
        for keep in (1, max(1, m // 4)):                                     # Ky Fan: the leading block is optimal
            assert abs(cv.captured_energy(a[b], v[b][:, :keep]) - want[:keep].sum()) < 1e-4 * top


@pytest.mark.parametrize('m,batch', [(3, 2), (66, 2), (97, 1), (127, 2), (1, 2), (2, 3), (5, 400), (16, 300), (59, 3)])
def test_symmetric_eigendecomposition_of_odd_orders(m, batch):
    # odd orders get an index of zeros, odd numbers of pairs split the triangle of blocks unevenly, small orders take fewer warps
    gu.ensure_built()
    rng = np.random.default_rng(130 + m)
    x = rng.standard_normal((batch, 3 * m + 2, m)) * (np.arange(1, m + 1) ** -0.7)
    a = np.einsum('bni,bnj->bij', x, x).astype(np.float32)
    w = torch.empty(batch, m, device='cuda'); v = torch.empty(batch, m, m, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    binding.transmla_conv_sym_eig(_dev(a), w, v, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    w, v = _f64(w), _f64(v)
    for b in range(batch):
        want, _ = cv.sorted_eigh(a[b])
        # bounds as for the even orders: at most 10 (m - 1) fp32 rotations of a column
        assert np.abs(w[b] - want).max() < 2e-5 * want[0]
        assert np.abs(v[b].T @ v[b] - np.eye(m)).max() < 1e-4
        assert np.abs(a[b].astype(np.float64) @ v[b] - v[b] * w[b]).max() < 1e-4 * want[0]


@pytest.mark.parametrize('fold', [1, 2])
def test_rorope_apply_matches_the_oracle_and_keeps_the_rope_inner_product(fold):
    gu.ensure_built()
    rng = np.random.default_rng(40)
    g, d, C = 4, 16, 70
    X = rng.standard_normal((g * d, C)).astype(np.float32)
    U = np.stack([np.linalg.qr(rng.standard_normal((g * fold, g * fold)))[0] for _ in range(d // 2 // fold)]).astype(np.float32)
    Y = torch.full((g * d, C), float('nan'), device='cuda')
    binding.transmla_conv_rorope_apply(_dev(X), _dev(U), g, d, fold, Y)
    want = cv.rorope_apply(X, U, g, d, fold)
    assert _rel(_f64(Y), want) < 1e-6
    if fold == 1:   # Eq. 18 on the CUDA result: columns 0 and 1 as a query and a key
        def merged_rope(x, pos):
            return orc.rope(x.reshape(g, d), pos).reshape(-1)
        y = _f64(Y)
        for t, j in [(3, 1), (900, 17)]:
            want_ip = merged_rope(X[:, 0].astype(np.float64), t) @ merged_rope(X[:, 1].astype(np.float64), j)
            got_ip = merged_rope(y[:, 0], t) @ merged_rope(y[:, 1], j)
            assert abs(got_ip - want_ip) < 1e-4 * max(1.0, abs(want_ip))


@pytest.mark.parametrize('g,d,fold,C', [(32, 128, 4, 192), (3, 16, 4, 68), (5, 4, 2, 65), (1, 2, 1, 3), (8, 8, 1, 1028),
                                        (9, 4, 1, 515), (16, 8, 2, 260), (33, 4, 1, 129), (65, 2, 1, 66)])
def test_rorope_apply_at_the_edges_of_its_tiles(g, d, fold, C):
    # the largest order, orders off the 8 values of a thread, columns off the tile of 64 and off the 4 of a thread
    gu.ensure_built()
    rng = np.random.default_rng(41)
    X = rng.standard_normal((g * d, C)).astype(np.float32)
    U = rng.standard_normal((d // 2 // fold, g * fold, g * fold)).astype(np.float32)
    Y = torch.full((g * d, C), float('nan'), device='cuda')
    binding.transmla_conv_rorope_apply(_dev(X), _dev(U), g, d, fold, Y)
    assert _rel(_f64(Y), cv.rorope_apply(X, U, g, d, fold)) < 1e-6     # at most 128 fp32 roundings that average out


def test_alpha_and_balanced_concatenation():
    gu.ensure_built()
    rng = np.random.default_rng(50)
    n, mk, mv = 1000, 48, 64
    k = (3.0 * rng.standard_normal((n, mk))).astype(np.float32)
    v = rng.standard_normal((n, mv)).astype(np.float32)
    alpha = torch.zeros(1, device='cuda')
    scratch = torch.empty(2 * n, device='cuda')
    binding.transmla_conv_alpha(_dev(k), _dev(v), scratch, alpha)
    want = cv.bkv_alpha(k, v)
    assert abs(float(alpha.item()) - want) < 1e-5 * want
    Z = torch.full((n, mk + mv), float('nan'), device='cuda')
    binding.transmla_conv_balance_concat(_dev(k), _dev(v), alpha, Z)
    z = _f64(Z)
    assert _rel(z[:, :mk], k.astype(np.float64) / float(alpha.item())) < 1e-6 and np.array_equal(z[:, mk:], v.astype(np.float64))


@pytest.mark.parametrize('n,mk,mv', [(1, 1, 1), (700, 4, 8), (5000, 16, 16), (333, 5, 2), (3, 3968, 4096), (129, 1001, 24)])
def test_concatenation_of_short_and_long_rows(n, mk, mv):
    # from one thread a row to a block a row, rows that are and are not whole 16 bytes
    gu.ensure_built()
    k, v = torch.randn(n, mk, device='cuda'), torch.randn(n, mv, device='cuda')
    alpha = torch.tensor([1.7], device='cuda')
    z = torch.full((n, mk + mv), float('nan'), device='cuda')
    binding.transmla_conv_balance_concat(k, v, alpha, z)
    assert torch.equal(z, torch.cat([k * (1.0 / alpha), v], dim=1))


@pytest.mark.parametrize('m,r', [(96, 24), (300, 64), (333, 33), (40, 1), (200, 129), (1100, 1024)])
def test_top_subspace_captures_what_the_leading_eigenvectors_capture(m, r):
    gu.ensure_built()
    # (orders that do and do not fill the factor's blocks of 32, up to the largest)
    rng = np.random.default_rng(60 + m)
    basis = np.linalg.qr(rng.standard_normal((m, m)))[0]
    lam = np.concatenate([np.linspace(50.0, 10.0, r), np.linspace(4.0, 0.01, m - r)])   # a clear gap after r
    Cm = ((basis * lam) @ basis.T).astype(np.float32)
    Q = _dev(rng.standard_normal((m, r)))
    scratch = torch.empty(binding.transmla_conv_subspace_scratch_bytes(m, r), dtype=torch.uint8, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    binding.transmla_conv_top_subspace(_dev(Cm), Q, 25, scratch, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    q = _f64(Q)
    assert np.abs(q.T @ q - np.eye(r)).max() < 1e-4
    vals, R = cv.joint_pca(np.linalg.cholesky(Cm.astype(np.float64) + 1e-9 * np.eye(m)).T, r)   # Z with Z^T Z = C
    assert cv.captured_energy(Cm, q) >= (1 - 1e-4) * vals[:r].sum()
    assert np.linalg.norm(q @ q.T - R @ R.T) < 1e-2 * np.sqrt(r)      # the same subspace (projectors agree)


@pytest.mark.parametrize('most', [1, 2, 4, 8])
@pytest.mark.parametrize('m,r', [(400, 70), (700, 512), (1100, 1024)])
def test_the_factor_in_smaller_clusters(m, r, most):
    # a CTA then owns more blocks of a panel than it holds at once; every block is the same sum in the same order
    gu.ensure_built()
    rng = np.random.default_rng(90 + m)
    x = rng.standard_normal((2 * m, m)) * np.arange(1, m + 1) ** -0.5
    C, q0 = _dev(x.T @ x), _dev(rng.standard_normal((m, r)))
    scratch = torch.empty(binding.transmla_conv_subspace_scratch_bytes(m, r), dtype=torch.uint8, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    full, part = q0.clone(), q0.clone()
    binding.transmla_conv_top_subspace(C, full, 2, scratch, status)
    binding.transmla_selftest_conv_subspace(C, part, 2, scratch, most, status)
    assert int(status.item()) == 0 and torch.equal(full, part)


@pytest.mark.parametrize('m,r', [(1000, 128), (700, 33), (600, 301), (50, 1)])
def test_the_basis_is_orthonormal_to_one_rounding_an_element(m, r):
    # rounding q_i and q_j to fp32 moves their product by 2 x 2^-24 at most (the pass itself works in fp64 or on differences)
    gu.ensure_built()
    rng = np.random.default_rng(80 + m)
    x = rng.standard_normal((2 * m, m)) * np.arange(1, m + 1) ** -0.5
    Q = _dev(rng.standard_normal((m, r)))
    scratch = torch.empty(binding.transmla_conv_subspace_scratch_bytes(m, r), dtype=torch.uint8, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    binding.transmla_conv_top_subspace(_dev(x.T @ x), Q, 5, scratch, status)
    q = _f64(Q)
    assert int(status.item()) == 0 and np.abs(q.T @ q - np.eye(r)).max() < 2.0 ** -23


def test_inverse_root_of_the_factor_over_all_exponents():
    # The result's roundings: d y by 2^-53, e by 2^-54 more, half of which reaches the result, and the last one 2^-53; the method
    # leaves 5/16 e^3, which an approximation to 2^-18 would bring to 2^-52.7 and the one there is (2^-20) to 2^-58.
    gu.ensure_built()
    rng = np.random.default_rng(95)
    mant = np.concatenate([[1.0, np.nextafter(1, 2), np.nextafter(2, 1), 1.5], 1 + rng.random(60)])
    d = np.ldexp(mant[None, :], np.arange(-1022, 1024)[:, None]).ravel()
    out = torch.empty(d.size, 3, dtype=torch.float64, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    binding.transmla_selftest_conv_inverse_root(torch.tensor(d, device='cuda'), out, status)
    got = out.cpu().numpy().astype(np.longdouble)
    off = np.abs(got * np.sqrt(d.astype(np.longdouble))[:, None] - 1).max(axis=0)
    assert int(status.item()) == 0
    assert off[0] <= 2.0 ** -52 and off[1] <= 2.0 ** -52 and off[2] <= 2.0 ** -20, np.log2(off.astype(np.float64))
    for bad in (0.0, -0.0, -1.0, np.nan, -np.inf):
        status.zero_()
        binding.transmla_selftest_conv_inverse_root(torch.tensor([bad], dtype=torch.float64, device='cuda'), out, status)
        assert int(status.item()) == 8 and float(out[0, 0]) == 1.0, bad       # TRANSMLA_DEV_NUMERIC
    binding.transmla_selftest_conv_inverse_root(torch.tensor([np.inf], dtype=torch.float64, device='cuda'), out, status)
    assert not np.isfinite(float(out[0, 0]))                                  # which the next pivot or pass reports


@pytest.mark.parametrize('m,r', [(100, 1), (200, 33), (200, 64), (300, 70), (600, 301), (1100, 1024)])
@pytest.mark.parametrize('what', [0.0, float('nan'), float('inf')])
def test_a_basis_without_full_rank_is_reported(m, r, what):
    # a column of zeros, and one value that is not finite, in the first column, inside a step of four and in the last column
    gu.ensure_built()
    rng = np.random.default_rng(96)
    x = rng.standard_normal((2 * m, m))
    C, q0 = _dev(x.T @ x), _dev(rng.standard_normal((m, r)))
    scratch = torch.empty(binding.transmla_conv_subspace_scratch_bytes(m, r), dtype=torch.uint8, device='cuda')
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    for column in sorted({0, r // 2, r - 1}):
        q = q0.clone()
        q[slice(None) if what == 0.0 else 5, column] = what
        status.zero_()
        binding.transmla_conv_top_subspace(C, q, 1, scratch, status)
        assert int(status.item()) & 8, column                                 # TRANSMLA_DEV_NUMERIC
    status.zero_()
    binding.transmla_conv_top_subspace(C, q0, 1, scratch, status)
    assert int(status.item()) == 0 and bool(torch.isfinite(q0).all())


def test_whole_conversion_step_by_step_against_the_oracle():
    # activations -> per-group covariances -> rotations -> rotated W_K -> alpha -> joint second moment -> basis -> rewrite
    gu.ensure_built()
    n, D, g, d, fold, r = 600, 96, 4, 16, 2, 40
    case = synth.make_conversion_case(n, D, g, d, seed=70, device='cuda')
    x, w_k, w_v = case['x'], case['w_k'], case['w_v']
    status = torch.zeros(1, dtype=torch.int32, device='cuda')
    k_act = torch.empty(n, g * d, device='cuda')
    binding.transmla_conv_gemm(x, w_k, k_act, tb=True)                       # k_t = W_K x_t
    assert _rel(_f64(k_act), _f64(x) @ _f64(w_k).T) < 1e-5
    groups, m = d // 2 // fold, g * fold
    cov = torch.empty(groups, m, m, device='cuda')
    scratch = torch.empty(binding.transmla_conv_rorope_scratch_bytes(n, g, d, fold) // 4, device='cuda')
    binding.transmla_conv_rorope_covariance(k_act, g, d, fold, scratch, cov)
    assert _rel(_f64(cov), cv.rorope_covariances(_f64(k_act), g, d, fold)) < 1e-5
    vals = torch.empty(groups, m, device='cuda'); U = torch.empty(groups, m, m, device='cuda')
    binding.transmla_conv_sym_eig(cov.clone(), vals, U, status)
    want_vals, _ = cv.rorope_rotations(_f64(cov))
    assert np.abs(_f64(vals) - want_vals).max() < 2e-5 * want_vals.max()
    # Prop. 2 on the CUDA eigenvalues: folding keeps at least what separate rotations keep
    cov1 = torch.empty(d // 2, g, g, device='cuda')
    s1 = torch.empty(binding.transmla_conv_rorope_scratch_bytes(n, g, d, 1) // 4, device='cuda')
    binding.transmla_conv_rorope_covariance(k_act, g, d, 1, s1, cov1)
    v1 = torch.empty(d // 2, g, device='cuda'); u1 = torch.empty(d // 2, g, g, device='cuda')
    binding.transmla_conv_sym_eig(cov1, v1, u1, status)
    for G in range(groups):
        assert float(vals[G, :fold].sum()) >= float(v1[G * fold:(G + 1) * fold, 0].sum()) * (1 - 1e-5)
    # rotate W_K with the CUDA rotations; the oracle does the same step with the same U
    w_k_rot = torch.empty_like(w_k)
    binding.transmla_conv_rorope_apply(w_k, U, g, d, fold, w_k_rot)
    assert _rel(_f64(w_k_rot), cv.rorope_apply(_f64(w_k), _f64(U), g, d, fold)) < 1e-5
    # head 0 keeps RoPE; heads 1.. are the NoPE keys (Sec. 4.3)
    w_k_nope = w_k_rot[d:].contiguous()
    k_nope = torch.empty(n, (g - 1) * d, device='cuda'); v_act = torch.empty(n, g * d, device='cuda')
    binding.transmla_conv_gemm(x, w_k_nope, k_nope, tb=True)
    binding.transmla_conv_gemm(x, w_v, v_act, tb=True)
    alpha = torch.zeros(1, device='cuda'); ns = torch.empty(2 * n, device='cuda')
    binding.transmla_conv_alpha(k_nope, v_act, ns, alpha)
    want_alpha = cv.bkv_alpha(_f64(k_nope), _f64(v_act))
    assert abs(float(alpha.item()) - want_alpha) < 1e-5 * want_alpha
    mz = (2 * g - 1) * d
    Z = torch.empty(n, mz, device='cuda')
    binding.transmla_conv_balance_concat(k_nope, v_act, alpha, Z)
    Cm = torch.empty(mz, mz, device='cuda')
    binding.transmla_conv_gemm(Z, Z, Cm, ta=True)
    assert _rel(_f64(Cm), _f64(Z).T @ _f64(Z)) < 1e-5
    gen = torch.Generator(device='cuda'); gen.manual_seed(71)
    Q = torch.randn(mz, r, generator=gen, device='cuda')
    ws = torch.empty(binding.transmla_conv_subspace_scratch_bytes(mz, r), dtype=torch.uint8, device='cuda')
    binding.transmla_conv_top_subspace(Cm, Q, 60, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    w_top, R = cv.joint_pca(_f64(Z), r)
    assert cv.captured_energy(_f64(Cm), _f64(Q)) >= (1 - 2e-3) * w_top[:r].sum()
    # rewrite (App. D.2 step 3) with the CUDA basis, against the oracle's rewrite with the same basis
    w_dkv = torch.cat([w_k_nope / alpha, w_v], dim=0).contiguous()           # [mz, D]
    w_ukv = torch.randn(50, mz, generator=gen, device='cuda')
    d2 = torch.empty(r, D, device='cuda'); u2 = torch.empty(50, r, device='cuda')
    binding.transmla_conv_gemm(Q, w_dkv, d2, ta=True)
    binding.transmla_conv_gemm(w_ukv, Q, u2)
    want_d, want_u = cv.low_rank_rewrite(_f64(w_dkv), _f64(w_ukv), _f64(Q))
    assert _rel(_f64(d2), want_d) < 1e-5 and _rel(_f64(u2), want_u) < 1e-5
    # what the compressed layer loses is what the oracle's own basis loses, to within the iteration's tolerance
    full = _f64(w_ukv) @ _f64(w_dkv) @ _f64(x).T
    err_cuda = np.linalg.norm(_f64(u2) @ (_f64(d2) @ _f64(x).T) - full)
    od, ou = cv.low_rank_rewrite(_f64(w_dkv), _f64(w_ukv), R)
    err_orc = np.linalg.norm(ou @ (od @ _f64(x).T) - full)
    assert err_cuda <= 1.05 * err_orc + 1e-6 * np.linalg.norm(full)
