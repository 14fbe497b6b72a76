"""Transforms and products over the whole range of prime sizes and ring sizes, against the CPU oracle, bit for bit.

The transforms keep lazy residues with rules that depend on the prime (below 2^55, below 2^57, larger; down to the
smallest size of 33 bits) and split the stages by ring size: the sizes around each rule, inputs at the ends
of the residue range (0 and q - 1, which drive the lazy bounds furthest) and random ones.
"""
import numpy as np
import pytest

import oracle
from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu

BITS = [33, 34, 40, 53, 54, 55, 55, 56, 56, 57, 57, 58, 59, 60, 60]


def pair(log_n, q_bits, p_bits, alpha, log_scale=32):
    args = (log_n, q_bits, p_bits, alpha, log_scale, 0, 1)
    return hedap.Context(*args), oracle.Context(*args)


@pytest.mark.parametrize("log_n", [10, 11, 12, 13, 14, 15, 16, 17])
def test_transforms_over_prime_sizes(log_n):
    bits = BITS if log_n <= 12 else [33, 55, 57, 60]
    g, o = pair(log_n, bits, [60, 60], 2)
    primes = o.primes()
    n = o.N
    top = np.stack([np.full(n, int(q) - 1, dtype=np.uint64) for q in primes])
    alt = top * (np.arange(n, dtype=np.uint64) & np.uint64(1))
    for x in (inputs.random_limbs(5, primes, n), top, alt, np.zeros_like(top)):
        fwd, inv = g.ntt(x, 0), g.ntt(x, 0, inverse=True)
        for i in range(len(primes)):
            assert np.array_equal(fwd[i], o.ntt(x[i], i)), (i, bits + [60, 60])
            assert np.array_equal(inv[i], o.ntt(x[i], i, inverse=True)), (i, bits + [60, 60])


@pytest.mark.parametrize("q_bits,p_bits,alpha", [
    ([60, 34, 57, 45, 55, 60], [60], 1),          # one prime a digit: nothing folded, one special prime
    ([60, 34, 57, 45, 55, 60, 40], [60, 60], 2),  # last limb added as it is or reduced
    ([60, 34, 57, 45, 55, 60, 40], [60] * 3, 3),  # a ragged last digit
    ([60, 34, 57, 45, 55, 60, 40], [60] * 5, 4),  # more than three products a word
    ([60, 34, 57, 45, 55, 60, 40, 56, 50], [60] * 8, 8),
])
def test_products_over_prime_sizes(q_bits, p_bits, alpha):
    g, o = pair(10, q_bits, p_bits, alpha)
    primes = o.primes()
    for level in range(1, len(q_bits)):
        for seed in (1, None):
            if seed is None:  # every word q - 1
                x = np.stack([np.stack([np.full(o.N, int(primes[i]) - 1, dtype=np.uint64) for i in range(level + 1)])] * 2)
            else:
                x = inputs.random_ciphertext_limbs(10 + level, primes, level, o.N)
            ga, oa = g.ct_import(x, level, o.scale), o.ct_import(x, level, o.scale)
            for op in ("mul", "mul_relin"):
                assert np.array_equal(getattr(g, op)(ga, ga).limbs(), getattr(o, op)(oa, oa).limbs()), (op, level)
            assert np.array_equal(g.rescale(ga).limbs(), o.rescale(oa).limbs()), level
            assert np.array_equal(g.rotate(ga, 3).limbs(), o.rotate(oa, 3).limbs()), level


def test_transform_of_device_words_at_an_odd_word():
    """Device arrays need 8-byte alignment only: a view that starts at an odd word transforms like an aligned one."""
    import torch
    g = hedap.Context(11, [45, 45, 45], [60], 1, 40.0, 0, 1)
    primes = g.primes()
    x = torch.from_numpy(inputs.random_limbs(3, np.tile(primes[:3], 2), g.N).astype(np.int64)).cuda()
    for inverse in (False, True):
        want = g.ntt_batch(x.clone(), 3, 0, inverse=inverse)
        buf = torch.empty(x.numel() + 1, dtype=torch.int64, device="cuda")
        odd = buf[1:].view(x.shape)
        odd.copy_(x)
        assert odd.data_ptr() % 16 == 8
        assert torch.equal(g.ntt_batch(odd, 3, 0, inverse=inverse), want)
        odd.copy_(x)
        assert torch.equal(g.ntt(odd[:3], 0, inverse=inverse), want[:3])
