"""Sizes at which a kernel's tiling or a dispatch rule changes, through the public calls, against the oracle.

The bars are those of the FP64 solver: eigenvalues to 1e-10 relative, principal angles to 1e-8; a product to 1e-12 of each
column's largest entry.
"""
import numpy as np
import pytest

import oracle as O
from paper_1512_06500_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_06500_gb300 import build_lib, eda as E
    build_lib.build()
    E.load()
    return E


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


# block widths around the register slices of the Cholesky factorisation with inverse (32, 64, 96 columns) and of one
# warp's rows (8); the wide ones exceed the rank of the problem, so pivots are lost and refilled
@pytest.mark.parametrize("b", [1, 7, 8, 9, 31, 32, 33, 64, 65, 96, 97])
def test_solve_block_width_edges(eda, b):
    p = synth.gaussian_clusters(d=700, k=9, n_per_class=[3, 4, 5, 3, 4, 5, 3, 4, 5], seed=77)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(block_b=b, tau=8.0)) as h:
        V, lam, _, info, code = h.solve(p.k - 1, 1e-11)
        assert code == 0, info
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=h.c2, tier="projected")
    V = V.cpu().numpy().T
    assert np.abs(V.T @ V - np.eye(p.k - 1)).max() <= 1e-13
    assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
    assert O.sin_angle(ref["V"], V) <= 1e-8


# block products with few inner rows, from the row count on at which a warp takes them whole (rows / 32 times blocks of 8
# columns >= 608 warps, up to 64 inner rows), just below it and beyond 64
@pytest.mark.parametrize("d,b", [(4831, 32), (4865, 32), (9001, 17), (2600, 64), (2600, 65)])
def test_solve_block_products(eda, d, b):
    p = synth.gaussian_clusters(d=d, k=20, n_per_class=5, seed=b)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(block_b=b, tau=8.0)) as h:
        V, lam, _, info, code = h.solve(p.k - 1, 1e-11)
        assert code == 0, info
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=h.c2, tier="projected")
    V = V.cpu().numpy().T
    assert np.abs(V.T @ V - np.eye(p.k - 1)).max() <= 1e-13
    assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
    assert O.sin_angle(ref["V"], V) <= 1e-8


# matrix orders around the eigensolver's rules (cluster sizes double from 24 columns on, the cooperative grid starts at
# 288, one exchange chunk holds 512 rows, the columns of 608 and more no longer come four to a CTA) and its smallest
@pytest.mark.parametrize("n", [2, 3, 4, 5, 23, 24, 25, 48, 97, 192, 257, 287, 288, 289, 511, 513, 609, 700])
def test_gram_eigenvalue_orders(eda, n):
    rng = np.random.default_rng(n)
    d = 720
    k = max(1, n // 6)
    lab = rng.permutation(np.arange(n) % k).astype(np.int32)
    X = rng.random((n, d))
    with eda.build(_dev(X), _dev(lab), k, eda.config(tau=5.0)) as h:
        f = h.factors()
        c2 = h.c2
    G = f["GW"].cpu().numpy()
    ev, Q = np.linalg.eigh(G)
    # Householder reduction and bisection are backward stable: errors of order n eps ||G||
    assert np.abs(f["evals_w"].cpu().numpy() - ev).max() <= 4 * n * np.finfo(float).eps * ev[-1]
    z = -0.5 * c2 * np.maximum(ev, 0.0)
    phi = np.where(z == 0.0, 1.0, np.expm1(z) / np.where(z == 0.0, 1.0, z))
    K = (Q * (-0.5 * c2 * phi)) @ Q.T
    assert np.abs(f["KW"].cpu().numpy() - K).max() <= 1e-11 * np.abs(K).max()


# the same reduction with the columns in a global slab: the largest Gram of a batch, whose kernels share the GPU
def test_batched_large_gram(eda):
    ps = [synth.gaussian_clusters(d=900, k=9, n_per_class=nj, seed=40 + nj) for nj in (72, 30, 20)]
    probs = [dict(X=_dev(p.X), labels=_dev(p.labels), k=p.k, t=p.k - 1, tol=1e-11) for p in ps]
    res, code = eda.solve_batched(probs, eda.config(block_b=8, tau=8.0), workers=3)
    assert code == 0
    for p, r in zip(ps, res):
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=r["info"]["c2"], tier="projected")
        assert np.max(np.abs(r["lam"].cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
        assert O.sin_angle(ref["V"], r["V"].cpu().numpy().T) <= 1e-8


# narrow symmetric products: widths around the three instances (8, 16, 32 columns) and the powers of two of the row phases,
# lengths around one CTA's rows and chunks, in FP64 (Grams) and single precision (the solver's block Grams)
@pytest.mark.parametrize("d,k", [(5, 2), (63, 3), (64, 4), (65, 5), (129, 8), (255, 9), (256, 16), (257, 17), (1000, 23),
                                 (4097, 31), (20011, 32), (20011, 33)])
def test_narrow_gram(eda, d, k):
    p = synth.gaussian_clusters(d=d, k=k, n_per_class=2, seed=d + k)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(tau=5.0)) as h:
        f = h.factors()
    for H, G in ((f["HB"], f["GB"]), (f["HW"], f["GW"])):
        H = H.cpu().numpy()
        G = G.cpu().numpy()
        assert np.array_equal(G, G.T)
        # a dot product of length d: |error| <= d eps sum |a||b|
        assert np.all(np.abs(G - H @ H.T) <= d * np.finfo(float).eps * (np.abs(H) @ np.abs(H).T) + 1e-300)


@pytest.mark.parametrize("b", [3, 8, 13, 16, 29, 32])
def test_narrow_block_single_precision(eda, b):
    p = synth.gaussian_clusters(d=1500, k=20, n_per_class=4, seed=b)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(prec=eda.EDA_F32, block_b=b, tau=6.0)) as h:
        V, lam, _, info, code = h.solve(p.k - 1, 1e-9)
        assert code == 0, info
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=h.c2, tier="projected")
    assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-9
    assert O.sin_angle(ref["V"], V.cpu().numpy().T) <= 1e-6


# blocks whose Gram loses a column to rounding without its pivot being recognised as lost: the new direction has to come out
# orthogonal to the basis all the same, whichever side of the threshold the rounding falls
@pytest.mark.parametrize("prec_name", ["f64", "tc"])
@pytest.mark.parametrize("seed,b", [(55, 3), (55, 4), (55, 5), (55, 7), (58, 3), (59, 3), (61, 5)])
def test_nearly_dependent_blocks(eda, seed, b, prec_name):
    p = synth.gaussian_clusters(d=333, k=7, n_per_class=[2, 3, 5, 1, 4, 3, 2], seed=seed)
    prec = eda.EDA_F64 if prec_name == "f64" else eda.EDA_F64_TC
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(prec=prec, block_b=b, tau=8.0, tc_min_mi=-1)) as h:
        ref = O.eda(p.X, p.labels, p.k, 6, c2=h.c2, tier="projected")
        for V, lam, code in ((lambda r: (r[0], r[1], r[3]))(h.solve_arnoldi(6, 1e-12)),
                             (lambda r: (r[0], r[1], r[4]))(h.solve(6, 1e-12))):
            assert code == 0
            assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
            assert O.sin_angle(ref["V"], V.cpu().numpy().T) <= 1e-8


# tensor-core FP64 products with more than 32 right-hand sides (one launch over all 32-column blocks): the edges of a block
# and of a 128-row band, K splits on and off, and an operand with room for more columns than it holds (the Krylov basis)
@pytest.mark.parametrize("d,k,nj,b", [(1000, 34, 3, 8), (4097, 66, 2, 16), (700, 65, 4, 33), (9000, 45, 12, 40)])
def test_wide_right_hand_sides(eda, d, k, nj, b):
    p = synth.gaussian_clusters(d=d, k=k, n_per_class=nj, seed=d + k)
    cfg = eda.config(prec=eda.EDA_F64_TC, block_b=b, tau=8.0, tc_min_mi=-1)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, cfg) as h:
        rng = np.random.default_rng(k)
        f = O.scatter_factors(p.X, p.labels, p.k)
        for m in (33, 64, 65, 129):
            X = rng.standard_normal((d, m))
            Y = h.apply_exp(eda.OP_M, _dev(X.T)).cpu().numpy().T
            Yr = O.m_apply(f["HW"], f["HB"], h.c2, X)
            assert (np.abs(Y - Yr).max(0) <= 1e-12 * np.abs(Yr).max(0)).all()
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=h.c2, tier="projected")
        for V, lam, code in ((lambda r: (r[0], r[1], r[4]))(h.solve(p.k - 1, 1e-11)),
                             (lambda r: (r[0], r[1], r[3]))(h.solve_direct(p.k - 1))):
            assert code == 0
            V = V.cpu().numpy().T
            assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
            assert O.sin_angle(ref["V"], V) <= 1e-8
            assert np.abs(V.T @ V - np.eye(p.k - 1)).max() <= 1e-12


# the stacked [G_W; G_BW] operand (from n = 512 on) and the split G_WB (from n k = 2^18 entries on) of the composed M-apply,
# on either side of both rules
@pytest.mark.parametrize("k,nj", [(64, 8), (85, 6), (255, 4), (256, 4)])
def test_composed_m_apply_operands(eda, k, nj):
    p = synth.gaussian_clusters(d=1300, k=k, n_per_class=nj, seed=k)
    f = O.scatter_factors(p.X, p.labels, p.k)
    rng = np.random.default_rng(k)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(prec=eda.EDA_F64_TC, tau=8.0, tc_min_mi=-1)) as h:
        for m in (1, 32, 40):
            X = rng.standard_normal((1300, m))
            Y = h.apply_exp(eda.OP_M, _dev(X.T)).cpu().numpy().T
            Yr = O.m_apply(f["HW"], f["HB"], h.c2, X)
            assert (np.abs(Y - Yr).max(0) <= 1e-12 * np.abs(Yr).max(0)).all()


# narrow products with more 128-row bands than SMs (152), dealt to the CTAs in runs: of whole bands for short rows, even ones
# for longer (a run's pieces joined); bands of one row, one column and a full block of 32
@pytest.mark.parametrize("d,k,nj", [(19457, 8, 3), (19585, 66, 3), (40000, 40, 10)])
def test_narrow_product_runs(eda, d, k, nj):
    p = synth.gaussian_clusters(d=d, k=k, n_per_class=nj, seed=d)
    f = O.scatter_factors(p.X, p.labels, p.k)
    rng = np.random.default_rng(k)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(prec=eda.EDA_F64_TC, tau=8.0, tc_min_mi=-1)) as h:
        for m in (1, 32):
            X = rng.standard_normal((d, m))
            Y = h.apply_exp(eda.OP_M, _dev(X.T)).cpu().numpy().T
            Yr = O.m_apply(f["HW"], f["HB"], h.c2, X)
            assert (np.abs(Y - Yr).max(0) <= 1e-12 * np.abs(Yr).max(0)).all()


# eigenvectors through the back-transformation: matrix orders n - 1 around its smallest blocked size (64) and its blocks of 32
# reflectors, few and many columns (1 to 8 a CTA by the number of columns)
@pytest.mark.parametrize("n,t", [(34, 3), (64, 5), (65, 1), (66, 40), (67, 66), (98, 9), (99, 98), (131, 64), (400, 399)])
def test_direct_solve_orders(eda, n, t):
    k = max(2, n // 3)
    counts = [n // k + (1 if j < n % k else 0) for j in range(k)]
    p = synth.gaussian_clusters(d=1100, k=k, n_per_class=counts, seed=n)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(tau=6.0)) as h:
        V, lam, info, code = h.solve_direct(t)
        assert code == 0
        c2 = h.c2
        V = V.cpu().numpy().T
        MV = h.apply_exp(eda.OP_N, _dev(V.T)).cpu().numpy().T
    # beyond the k - 1 eigenvalues above 1 the direct solver's pairs are those of span[H_W H_B] (below 1), the oracle's t
    # largest the unit ones of its complement
    m = min(t, p.k - 1)
    ref = O.eda(p.X, p.labels, p.k, m, c2=c2, tier="projected")
    assert np.max(np.abs(lam.cpu().numpy()[:m] - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
    assert np.abs(V.T @ V - np.eye(t)).max() <= 1e-12
    # span(V) is invariant under N: N V = V (V^T N V) up to 1e-10 of ||N|| <= lambda_1 (the spectrum below may be close)
    assert np.abs(MV - V @ (V.T @ MV)).max() <= 1e-9 * ref["lam_t"][0]


# Gram matrices whose columns all but decouple: classes of two opposite samples in pixels of their own, with one pixel in
# common that couples them by 1e-60 and 1e-140 (squares of the coupling in range) and 1e-160 (out of range); cluster and grid
@pytest.mark.parametrize("k", [6, 40, 150, 170])
@pytest.mark.parametrize("c", [1e-30, 1e-70, 1e-80])
def test_gram_eigenvalues_tiny_couplings(eda, k, c):
    n, d = 2 * k, k + 40
    X = np.zeros((n, d))
    for j in range(k):
        X[2 * j, j] = 1.0 + j / k
        X[2 * j, d - 1] = c
        X[2 * j + 1] = -X[2 * j]
    lab = np.repeat(np.arange(k), 2).astype(np.int32)
    with eda.build(_dev(X), _dev(lab), k, eda.config(tau=2.0, c2=0.1)) as h:
        f = h.factors()
    G, ev = f["GW"].cpu().numpy(), f["evals_w"].cpu().numpy()
    ref = np.linalg.eigvalsh(G)
    assert np.abs(ev - ref).max() <= 4 * n * np.finfo(float).eps * ref[-1]


# Kernels launched to be set up while their predecessor runs: long chains of short ones (small and middle sizes, with and
# without chip-filling kernels between), with another stream keeping the SMs busy unevenly. All sums are taken in a fixed
# order, so a kernel that read before its predecessor had finished would show as different bits.
@pytest.mark.parametrize("mode,d,k,per", [("EDA_F64", 96, 4, 3), ("EDA_F64", 1500, 24, 5), ("EDA_F64_TC", 1500, 24, 5),
                                          ("EDA_BF16", 1500, 24, 5), ("EDA_F32", 700, 9, 4)])
def test_chained_launches_give_the_same_bits(eda, mode, d, k, per):
    p = synth.gaussian_clusters(d=d, k=k, n_per_class=[per] * k, seed=5)
    X, lab = _dev(p.X), _dev(p.labels)
    other = torch.cuda.Stream()
    busy = torch.randn(900, 900, device="cuda:0")
    with eda.build(X, lab, k, eda.config(tau=6.0, prec=getattr(eda, mode))) as h:
        first = None
        for i in range(6):
            if i % 2:
                with torch.cuda.stream(other):
                    for _ in range(60):
                        busy = torch.tanh(busy @ busy / 30.0)
            V, lam, _, _, code = h.solve(k - 1, 1e-9, check=False)
            assert code in (0, -8)
            if first is None:
                first = (V.clone(), lam.clone())
            assert torch.equal(V, first[0]) and torch.equal(lam, first[1])
        # recorded into a graph: replayed on inputs written after the capture
        x = torch.zeros(5, d, dtype=torch.float64, device="cuda:0")
        y = torch.empty_like(x)
        h.apply_exp(eda.OP_M, x, out=y)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            h.apply_exp(eda.OP_M, x, out=y, stream=torch.cuda.current_stream())
        x.copy_(torch.randn(5, d, dtype=torch.float64, device="cuda:0"))
        g.replay()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, h.apply_exp(eda.OP_M, x))
    torch.cuda.synchronize()
