"""Sums whose order is part of the result, and the resources a call may take."""
import subprocess
import sys
from fractions import Fraction

import numpy as np
import pytest

import synthetic_inputs as si
from tests.helpers import cuda_torch, gpu_lib, make_case

pytestmark = pytest.mark.gpu

FP64, BF16X3, FP64_TC = 0, 1, 4


def test_integrals_are_chains_of_fused_multiply_adds(tmp_path):
    """(pq|rs) formed on the device: one chain per integral, Cholesky vectors in order.

    Against the same integrals formed here (each step exact, rounded once) and given as
    the full array: diagonal and sigma agree to the bit."""
    torch = cuda_torch()
    g = gpu_lib()
    K, N, D, k = 8, 8, 40, 4
    h, L, _, path = make_case(tmp_path, K, N, 0, D, center=k)
    flat = L.reshape(L.shape[0], -1)
    exact = [[Fraction(float(x)) for x in row] for row in flat]
    n = K * K
    eri = np.zeros((n, n))
    for a in range(n):
        for b in range(a, n):
            s = 0.0
            for row in exact:
                s = float(row[a] * row[b] + Fraction(s))
            eri[a, b] = eri[b, a] = s
    out = []
    for chol in (L, eri.reshape(K, K, K, K)):
        plan = g.Plan(h, chol, K, N, 0, D, path, precision=FP64)
        plan.set_bond(k)
        psi = torch.from_numpy(si.random_vector(plan.dim, seed=1)).cuda()
        y, d = torch.empty_like(psi), torch.empty_like(psi)
        plan.sigma(psi, y)
        plan.hdiag(d)
        torch.cuda.synchronize()
        out.append((y.cpu().numpy(), d.cpu().numpy()))
        plan.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("K,D,width", [(14, 600, 1.0), (20, 500, 1.2)])
def test_first_products_fit_the_scratch_that_was_allowed(tmp_path, K, D, width):
    """Sectors of one to three states beside wide ones: a chunk's stored products stay
    within scratch_bytes.

    The renormalisation before the bond fills the scratch up to less than one product
    (at most 190 x 192 elements of two pieces, 146 KB), and with a chunk per term sigma
    needs no more; so a list of several full chunks may hold at most that much more."""
    cuda_torch()
    g = gpu_lib()
    k, room = 4, 4 << 20
    h, L, _, path = make_case(tmp_path, K, K, 0, D, center=k, split="gaussian", wn=width, ws=width)
    held = []
    for per_term in (0, 1):
        plan = g.Plan(h, L, K, K, 0, D, path, precision=BF16X3, scratch_bytes=room, sigma_per_term=per_term)
        plan.set_bond(k)
        st = plan.stats()
        held.append(st["device_bytes"])
        if not per_term:
            assert st["sigma_chunks"] > 1
        plan.close()
    assert held[0] <= held[1] + (256 << 10)


def test_davidson_calls_repeat_and_match_fp64(tmp_path):
    """Mixed Davidson on a short list: eight steps from a random vector, stopped unconverged.

    Such a call makes any figure of its vector out of the last place of a sum, and the
    FP64 additions of K-chunks come in an order that repeats, not in a fixed one: with the
    schedule of short lists 1 call in 16 falls out (6 of 72 from its first call), with that
    of long lists 1 in 4 (17 of 72).  Of 48 calls (six problems, eight each, every one
    against the vector that most of its problem's calls agree on) 3 and 12 are expected;
    7 may.  The energy is that of the vector in FP64 arithmetic: to 4.6e-5 of |H x|, the
    bound of the mixed sigma."""
    torch = cuda_torch()
    g = gpu_lib()
    K, D, k = 14, 600, 7
    out = 0
    for seed in (20, 27, 28, 30, 32, 39):
        h, L = si.make_integrals(K, 4 * K, seed=2 * seed)
        mps = si.random_mps(K, K, 0, si.bond_sectors(K, K, 0, D, "gaussian", 1.0, 1.0), center=k, seed=2 * seed + 1)
        path = str(tmp_path / f"mps_{seed}.bin")
        si.write_mps(path, mps)
        plan = g.Plan(h, L, K, K, 0, D, path, precision=BF16X3, tc_kchunk=1024)
        plan.set_bond(k)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(plan.dim, dtype=torch.float64, device="cuda", generator=gen)
        x /= x.norm()
        got = []
        for _ in range(8):
            y = x.clone()
            e, _, _ = plan.davidson(y, 1, tol=1e-10, max_iter=8)
            got.append(y)
        off = [sum(float((a - b).norm()) > 1e-9 for b in got) for a in got]
        out += min(off)
        hy = torch.empty_like(y)
        plan.sigma_fp64(y, hy)
        assert abs(e[0] - float(y @ hy)) <= 4.6e-5 * float(hy.norm())
        plan.close()
    print(f"{out} of 48 calls off")
    assert out <= 7


def test_short_and_long_lists_of_all_piece_counts(tmp_path):
    """Davidson's own schedule of short lists against the one of dmrg_sigma: two steps from
    a vector with every sector filled give Ritz values of the same matrix, each off by at
    most the bound of the mixed sigma (4.6e-5 of |H x|; one piece 3e-2)."""
    torch = cuda_torch()
    g = gpu_lib()
    for precision, bound in ((1, 4.6e-5), (2, 3e-2), (3, 1.5e-5)):
        for K, D, k, tile_n in ((8, 64, 2, 0), (10, 100, 5, 64), (14, 600, 7, 0)):
            h, L, _, path = make_case(tmp_path, K, K, 0, D, center=k, split="gaussian", wn=1.0, ws=1.0)
            plan = g.Plan(h, L, K, K, 0, D, path, precision=precision, sigma_tile_n=tile_n)
            plan.set_bond(k)
            y = torch.from_numpy(si.random_vector(plan.dim, seed=3)).cuda()
            hy = torch.empty_like(y)
            y /= y.norm()
            plan.sigma(y, hy)
            z = y.clone()
            e, _, _ = plan.davidson(z, 1, tol=1e-10, max_iter=1)  # the Ritz value of one vector: x H x
            assert abs(e[0] - float(y @ hy)) <= 2 * bound * float(hy.norm())
            e, _, _ = plan.davidson(z, 1, tol=1e-10, max_iter=2)
            plan.sigma(z, hy)
            assert abs(e[0] - float(z @ hy) / float(z @ z)) <= 2 * bound * float(hy.norm())
            plan.close()


@pytest.mark.parametrize("K,D,width", [(12, 300, 1.0), (20, 300, 1.2)])
def test_fp64_accurate_sigma_repeats(tmp_path, K, D, width):
    """FP64_TC: sums up to 16384 deep are one addition, twice that two, in either order."""
    torch = cuda_torch()
    g = gpu_lib()
    k = K // 2
    h, L, _, path = make_case(tmp_path, K, K, 0, D, center=k, split="gaussian", wn=width, ws=width)
    plan = g.Plan(h, L, K, K, 0, D, path, precision=FP64_TC)
    plan.set_bond(k)
    rng = np.random.default_rng(1)
    x = np.ldexp(rng.standard_normal(plan.dim), rng.integers(-45, 1, plan.dim))  # partial sums of unlike size
    x = torch.from_numpy(x).cuda()
    first = None
    for _ in range(12):
        y = torch.empty_like(x)
        plan.sigma(x, y)
        first = y if first is None else first
        assert torch.equal(y, first)
    plan.close()


@pytest.mark.parametrize("K,D,width", [(10, 60, 1.0), (14, 400, 1.2)])
def test_tile_shape_does_not_depend_on_the_way_to_a_bond(tmp_path, K, D, width):
    """A plan that has come through the chain and a new one at the same bond (same sectors)
    choose the same tile shape, and say the same of the candidates."""
    torch = cuda_torch()
    g = gpu_lib()
    h, L, _, path = make_case(tmp_path, K, K, 0, D, center=2, split="gaussian", wn=width, ws=width)
    plan = g.Plan(h, L, K, K, 0, D, path, precision=BF16X3)
    plan.set_bond(2)
    for k in range(2, K - 2):
        x = torch.from_numpy(si.random_vector(plan.dim, seed=k)).cuda()
        room = torch.zeros(8 * plan.dim + 65536, dtype=torch.float64, device="cuda")
        plan.decimate(x, 1, D, True, next_psi=room, next_cap=room.numel())
        plan.set_bond(k + 1)
        here = str(tmp_path / "here.bin")
        plan.save_mps(here)
        fresh = g.Plan(h, L, K, K, 0, D, here, precision=BF16X3)
        fresh.set_bond(k + 1)
        a, b = plan.stats(), fresh.stats()
        assert plan.dim == fresh.dim
        for name in ("sigma_tile_n", "sigma_kchunk", "tune_cand_ms"):
            assert a[name] == b[name], (k + 1, name)
        fresh.close()
    plan.close()


FIRST_CALLS = """
import sys, threading
import numpy as np, torch
import paper_2311_02854_gb300 as g
rng = np.random.default_rng(4)
A, B = (torch.from_numpy(rng.standard_normal(48 * 96)).cuda() for _ in range(2))
blocks = [(48, 48, 0, [(96, 0, 96, 0, 0, 48, 0, 1.0)])]
C = [torch.full((48 * 48,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(6)]
torch.cuda.synchronize()
start = threading.Barrier(6)
def run(i):
    st = torch.cuda.Stream()
    start.wait()
    for _ in range(20):
        g.grouped_gemm(4, blocks, A, B, C[i], stream=st)
ts = [threading.Thread(target=run, args=(i,)) for i in range(6)]
[t.start() for t in ts], [t.join() for t in ts]
want = A.view(48, 96) @ B.view(96, 48)
for c in C:
    assert torch.equal(c, C[0])
    assert float((c.view(48, 48) - want).norm() / want.norm()) < 1e-12
print("ok")
"""


def test_first_fp64_accurate_products_of_several_threads():
    """Each call has an error word of its own: nothing is set up by whoever comes first."""
    cuda_torch()
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[-2000:]


def test_a_new_plan_takes_back_what_grouped_products_keep(tmp_path):
    """The pool of dmrg_grouped_gemm keeps memory between calls, but not from a plan."""
    torch = cuda_torch()
    g = gpu_lib()
    h, L, _, path = make_case(tmp_path, 6, 6, 0, 20, center=3)

    def plan():
        g.Plan(h, L, 6, 6, 0, 20, path).close()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    n = 4096
    a, b, c = (torch.ones(n * n, dtype=torch.float64, device="cuda") for _ in range(3))
    free = plan()
    g.grouped_gemm(BF16X3, [(n, n, 0, [(n, 0, n, 0, 0, n, 0, 1.0)])], a, b, c)
    torch.cuda.synchronize()
    assert float(c[0]) == n
    assert torch.cuda.mem_get_info()[0] <= free - (100 << 20)  # the pieces of a and b: 128 MB
    assert plan() >= free - (16 << 20)


@pytest.mark.parametrize("K,D,k,n_roots", [(4, 8, 1, 1), (6, 20, 3, 2), (8, 64, 4, 1), (10, 100, 5, 3), (12, 300, 4, 1),
                                           (14, 600, 7, 1)])
def test_fp64_davidson_sums_in_chains(tmp_path, K, D, k, n_roots):
    """The sigma inside an FP64 Davidson call (one chain per element, parts of every size,
    chains cut at 16384: the last case sums to 40 000) against dmrg_sigma: one step from
    orthonormal vectors gives the eigenvalues of X H X^T.  A sum of n terms is off by at most
    n u of the sum of their magnitudes on either side; 1e-12 of |H x| holds that at n = 4000
    with room for the sums' cancellation, the bar of the FP64 tests.  Calls repeat."""
    torch = cuda_torch()
    g = gpu_lib()
    h, L, _, path = make_case(tmp_path, K, K, 0, D, center=k, split="gaussian", wn=1.0, ws=1.0)
    plan = g.Plan(h, L, K, K, 0, D, path, precision=FP64, n_roots=n_roots)
    plan.set_bond(k)
    n_roots = min(n_roots, plan.dim)
    x = np.linalg.qr(si.random_vector(plan.dim, seed=1, nvec=n_roots).reshape(n_roots, plan.dim).T)[0].T.copy()
    x = torch.from_numpy(x).cuda()
    hx = torch.empty_like(x)
    plan.sigma(x, hx, nvec=n_roots)
    want = torch.linalg.eigvalsh((x @ hx.T + hx @ x.T) / 2).cpu().numpy()
    got = []
    for _ in range(2):
        y = x.clone()
        e, _, _ = plan.davidson(y, n_roots, tol=1e-14, max_iter=1)
        got.append((e, y))
    assert np.abs(np.sort(got[0][0]) - want).max() <= 1e-12 * float(hx.norm(dim=1).max()) * n_roots
    assert np.array_equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    z = x.clone()
    e, _, _ = plan.davidson(z, n_roots, tol=1e-14, max_iter=6)
    plan.sigma(z, hx, nvec=n_roots)  # of Ritz vectors
    for i in range(n_roots):
        assert abs(e[i] - float(z[i] @ hx[i])) <= 1e-11 * float(hx[i].norm())
    plan.close()
