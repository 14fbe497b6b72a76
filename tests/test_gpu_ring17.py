"""Products, rescales and rotations at N = 2^17 against the CPU oracle, bit for bit: the column phase of 2^9 rows with every
fused load (one to three terms from shared memory, more from L2), primes of both lazy rules, a ragged last digit."""
import numpy as np
import pytest

import oracle
from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q_bits,p_bits,alpha", [
    ([60, 34, 57, 45], [60], 1),
    ([60, 34, 57, 45, 50], [60, 60], 2),
    ([60, 34, 57, 45], [60] * 3, 3),
    ([60, 34, 57, 45, 50], [60] * 4, 4),
])
def test_products_at_the_largest_ring(q_bits, p_bits, alpha):
    args = (17, q_bits, p_bits, alpha, 32, 0, 1)
    g, o = hedap.Context(*args), oracle.Context(*args)
    level = len(q_bits) - 1
    primes = o.primes()
    top = np.stack([np.stack([np.full(o.N, int(primes[i]) - 1, dtype=np.uint64) for i in range(level + 1)])] * 2)
    for x in (inputs.random_ciphertext_limbs(3, primes, level, o.N), top):
        ga, oa = g.ct_import(x, level, o.scale), o.ct_import(x, level, o.scale)
        assert np.array_equal(g.mul(ga, ga).limbs(), o.mul(oa, oa).limbs())
        assert np.array_equal(g.mul_relin(ga, ga).limbs(), o.mul_relin(oa, oa).limbs())
        assert np.array_equal(g.rescale(ga).limbs(), o.rescale(oa).limbs())
        assert np.array_equal(g.rotate(ga, 3).limbs(), o.rotate(oa, 3).limbs())
