"""The engines at the edges of their tiles, parts, boxes and splits.

Bounds, all fixed by the arithmetic:
* FP64 products: a sum of K terms and s segments is off by at most
  (K + s + 4) u sum |alpha a b| per element, u = 2^-53 (twice that here: numpy
  rounds too).
* Mixed sigma against FP64 arithmetic: operands and the first product are kept
  to 2^-17 (two pieces), 2^-9 (one) or 2^-25 (three) of each element, four of
  them in a term, and tensor memory truncates about 2^-23 per 16-deep step, at
  most 64 steps per sum in each of the two products: 4 * 2^-17 + 128 * 2^-23 =
  4.6e-5 (BF16X3), 128 * 2^-23 = 1.5e-5 (BF16X6); one piece is held to the 3e-2
  of the mixed tests.
* FP64_TC sigma: 1e-12, the bar of the FP64 path."""
import threading

import numpy as np
import pytest

import synthetic_inputs as si
from oracle.dmrg import Oracle
from oracle.hamiltonian import eri_from_cholesky
from tests.helpers import cuda_torch, gpu_lib, make_case, rel_err

pytestmark = pytest.mark.gpu

FP64, BF16X3, BF16, BF16X6, FP64_TC = 0, 1, 2, 3, 4


def _products(rng, shapes, pieces=False):
    """Blocks (m, n, [k, ...]) in random orientations and leading dimensions
    (multiples of 8 where the bf16 pieces want that): the block list, the operands,
    and each block's product and sum of |terms|."""
    blocks, a, b, want = [], [], [], []
    ao = bo = co = 0
    for m, n, ks in shapes:
        segs = []
        C, M = np.zeros((m, n)), np.zeros((m, n))
        for k in ks:
            at, bt = int(rng.integers(0, 2)), int(rng.integers(0, 2))
            A = rng.standard_normal((k, m) if at else (m, k))
            B = rng.standard_normal((n, k) if bt else (k, n))
            lda, ldb = (-(-X.shape[1] // 8) * 8 if pieces else X.shape[1] + int(rng.integers(0, 4)) for X in (A, B))
            alpha = float(rng.choice([1.0, -1.0] if pieces else [1.0, -1.0, 0.75]))
            for X, ld, out in ((A, lda, a), (B, ldb, b)):
                Y = np.full((X.shape[0], ld), 0.0 if pieces else np.nan)  # (no result of the FP64 units reads between rows)
                Y[:, :X.shape[1]] = X
                out.append(Y.ravel())
            oA, oB = A.T if at else A, B.T if bt else B
            C += alpha * (oA @ oB)
            M += abs(alpha) * (np.abs(oA) @ np.abs(oB))
            segs.append((k, ao, lda, at, bo, ldb, bt, alpha))
            ao += A.shape[0] * lda
            bo += B.shape[0] * ldb
        blocks.append((m, n, co, segs))
        want.append((co, m, n, C, M, sum(ks), len(ks)))
        co += m * n
    one = np.zeros(1)
    return blocks, np.concatenate(a or [one]), np.concatenate(b or [one]), co, want


EDGES = (1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 97)
FP64_SHAPES = {
    "parts": [(m, n, [k]) for m in EDGES for n, k in ((1, 65), (16, 16), (33, 17), (64, 1), (65, 33))],
    "one long sum": [(20, 20, [5001])],
    "long sums": [(m, m, [1500, 700, 3]) for m in (5, 33, 70)],
    "many segments": [(10, 14, [int(k) for k in 1 + np.arange(300) % 37])],
    "few and empty": [(1, 1, [1]), (40, 3, []), (3, 40, [2, 2])],
    "large": [(200, 131, [150, 64, 1])],
}


@pytest.mark.parametrize("name", FP64_SHAPES)
def test_fp64_products(name):
    torch = cuda_torch()
    g = gpu_lib()
    blocks, A, B, nc, want = _products(np.random.default_rng(11), FP64_SHAPES[name])
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    got = []
    for _ in range(2):
        dC = torch.full((nc,), np.nan, dtype=torch.float64, device="cuda")
        g.grouped_gemm(FP64, blocks, dA, dB, dC)
        got.append(dC.cpu().numpy())
    assert np.array_equal(got[0], got[1])  # sums in a fixed order
    dC = torch.full((nc,), np.nan, dtype=torch.float64, device="cuda")
    g.grouped_gemm_noalloc(blocks, dA, dB, dC)
    assert np.array_equal(got[0], dC.cpu().numpy())  # the same split and order without allocations
    for off, m, n, C, M, K, s in want:
        err = np.abs(got[0][off:off + m * n].reshape(m, n) - C)
        assert np.all(err <= 2 * (K + s + 4) * 2.0 ** -53 * M), (m, n, K)


@pytest.mark.parametrize("shift", [0, 1])
def test_operands_at_any_alignment(shift):
    """The splits read four elements at a time where the address allows it."""
    torch = cuda_torch()
    g = gpu_lib()
    blocks, A, B, nc, _ = _products(np.random.default_rng(5), [(65, 33, [17, 40]), (16, 24, [8])], pieces=True)
    out = []
    for sh in (0, shift):
        dA = torch.zeros(A.size + 1, dtype=torch.float64, device="cuda")[sh:sh + A.size]
        dB = torch.zeros(B.size + 1, dtype=torch.float64, device="cuda")[sh:sh + B.size]
        dA.copy_(torch.from_numpy(A))
        dB.copy_(torch.from_numpy(B))
        dC = torch.empty(nc, dtype=torch.float64, device="cuda")
        g.grouped_gemm(BF16X3, blocks, dA, dB, dC)
        out.append(dC.cpu().numpy())
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


def test_pieces_over_the_range_of_the_exponent():
    """x * 1 is the two pieces of x: 2^-16 of it anywhere in bf16's normal range,
    zeros stay zero, what is beyond the range or not finite stays not finite."""
    torch = cuda_torch()
    g = gpu_lib()
    rng = np.random.default_rng(2)
    x = np.concatenate([np.ldexp(1.0 + rng.random(2000), rng.integers(-90, 120, 2000)) * rng.choice([-1, 1], 2000),
                        [0.0, -0.0, 1.0, 1 + 2.0 ** -24, 1 + 2.0 ** -25, 1 - 2.0 ** -53, 2 - 2.0 ** -52]])
    bad = np.array([np.inf, -np.inf, np.nan, 1e300])
    v = np.concatenate([x, bad])
    dA = torch.zeros((v.size, 8), dtype=torch.float64, device="cuda")
    dA[:, 0] = torch.from_numpy(v).cuda()
    dB = torch.ones(8, dtype=torch.float64, device="cuda")
    dC = torch.empty(v.size, dtype=torch.float64, device="cuda")
    g.grouped_gemm(BF16X3, [(1, 1, i, [(1, 8 * i, 8, 0, 0, 8, 0, 1.0)]) for i in range(v.size)], dA, dB, dC)
    got = dC.cpu().numpy()
    assert np.all(np.abs(got[:x.size] - x) <= 2.0 ** -16 * np.abs(x))
    assert not np.isfinite(got[x.size:]).any()


def test_products_from_several_threads():
    """The products' device memory comes from one pool: calls from several threads
    on streams of their own give what one thread gives."""
    torch = cuda_torch()
    g = gpu_lib()
    sets = []
    for i, prec in enumerate((FP64, BF16X3, FP64_TC, FP64)):
        blocks, A, B, nc, _ = _products(np.random.default_rng(i), [(70 + i, 40, [33, 9]), (8, 100, [64])] * 6, pieces=True)
        dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
        ref = torch.empty(nc, dtype=torch.float64, device="cuda")
        g.grouped_gemm(prec, blocks, dA, dB, ref)
        sets.append((prec, blocks, dA, dB, ref))
    torch.cuda.synchronize()
    bad = []

    def work(prec, blocks, dA, dB, ref):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(10):
                c = torch.empty_like(ref)
                g.grouped_gemm(prec, blocks, dA, dB, c)
                st.synchronize()
                if not torch.equal(c, ref):
                    bad.append(prec)

    ts = [threading.Thread(target=work, args=s) for s in sets]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


# sector sizes at the middle bond: 17 | 32 36 | 34 | 65 | 100 and 12 | 129 and less
CHAINS = [(10, 74, 0.8), (8, 100, 0.8), (10, 150, 0.8), (10, 283, 0.8), (10, 500, 0.8), (12, 560, 0.8)]


@pytest.mark.parametrize("prec,bound", [(BF16X3, 5e-5), (BF16, 3e-2), (BF16X6, 1.5e-5)])
@pytest.mark.parametrize("K,D,w", CHAINS)
def test_mixed_sigma_sector_sizes(tmp_path, K, D, w, prec, bound):
    torch = cuda_torch()
    g = gpu_lib()
    h, L, mps, path = make_case(tmp_path, K, K, 0, D, center=K // 2, split="gaussian", wn=w, ws=w)
    kchunk = set()
    for _ in range(2):
        plan = g.Plan(h, L, K, K, 0, D, path, precision=prec)
        plan.set_bond(K // 2)
        kchunk.add(plan.stats()["sigma_kchunk"])
        if len(kchunk) == 1 and _ == 0:
            plan.close()
    assert len(kchunk) == 1  # the shape is a rule on sizes: the same every time
    dim, nvec = plan.dim, 3
    x = torch.from_numpy(si.random_vector(dim, seed=1, nvec=nvec).reshape(nvec, dim).copy()).cuda()
    y, one, z = torch.full_like(x, np.nan), torch.empty_like(x), torch.empty_like(x)
    plan.sigma(x, y, nvec=nvec)
    for v in range(nvec):
        plan.sigma(x[v], one[v])
        plan.sigma_fp64(x[v], z[v])
    torch.cuda.synchronize()
    y, one, z = y.cpu().numpy(), one.cpu().numpy(), z.cpu().numpy()
    plan.close()
    for v in range(nvec):
        assert rel_err(y[v], z[v]) <= bound, rel_err(y[v], z[v])
        assert rel_err(y[v], one[v]) <= 1e-12  # the same sums, added to the result in another order


@pytest.mark.parametrize("K,D,w", CHAINS[:5])
def test_fp64_engines_sector_sizes(tmp_path, K, D, w):
    """FP64 units and FP64_TC on the same problem, several vectors; the diagonal and,
    for the smaller problems, the result against the oracle."""
    torch = cuda_torch()
    g = gpu_lib()
    k, nvec = K // 2, 2
    h, L, mps, path = make_case(tmp_path, K, K, 0, D, center=k, split="gaussian", wn=w, ws=w)
    out, diag = {}, {}
    for prec in (FP64, FP64_TC):
        plan = g.Plan(h, L, K, K, 0, D, path, precision=prec)
        plan.set_bond(k)
        dim = plan.dim
        psi = si.random_vector(dim, seed=1, nvec=nvec).reshape(nvec, dim)
        x = torch.from_numpy(psi.copy()).cuda()
        y = torch.full_like(x, np.nan)
        d = torch.full((dim,), np.nan, dtype=torch.float64, device="cuda")
        plan.sigma(x, y, nvec=nvec)
        plan.hdiag(d)
        out[prec], diag[prec] = y.cpu().numpy(), d.cpu().numpy()
        plan.close()
    for v in range(nvec):
        assert rel_err(out[FP64_TC][v], out[FP64][v]) <= 1e-12
    if D <= 150:
        ts = Oracle(h, eri_from_cholesky(L), K, 0, mps).two_site(k)
        for v in range(nvec):
            assert rel_err(out[FP64][v], ts.sigma(psi[v])) <= 1e-12
        ref = ts.hdiag()
        for prec in diag:
            assert np.abs(diag[prec] - ref).max() <= 1e-11 * np.abs(ref).max()
