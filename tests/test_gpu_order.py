"""Sums whose order is part of the result, and the resources a call may take."""
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
