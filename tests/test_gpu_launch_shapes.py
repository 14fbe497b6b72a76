"""Every launch shape of the two-launch transforms against the CPU oracle, bit for bit: on a ring above the thread-block clusters'
(every transform there has a shape), and on the small rings with more words than those take (2^21) or with more than the
separate key inner product takes (2^18 a digit)."""
import numpy as np
import pytest

import oracle
from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu

SHAPES = (0, 1)  # variants of equal parity are one shape


def pair(log_n, q_bits, p_bits, alpha):
    args = (log_n, q_bits, p_bits, alpha, 32, 0, 1)
    return hedap.Context(*args), oracle.Context(*args)


@pytest.mark.parametrize("v", SHAPES)
def test_transforms_in_every_shape(v):
    g, o = pair(14, [33, 55, 57, 60], [60], 1)
    primes = o.primes()
    x = inputs.random_limbs(17, primes, o.N)
    g.ntt_set_variant(v, v)
    fwd, inv = g.ntt(x, 0), g.ntt(x, 0, inverse=True)
    for i in range(len(primes)):
        assert np.array_equal(fwd[i], o.ntt(x[i], i)), i
        assert np.array_equal(inv[i], o.ntt(x[i], i, inverse=True)), i


@pytest.mark.parametrize("q_bits,p_bits,alpha", [
    ([60, 34, 57, 45, 50], [60], 1),
    ([60, 34, 57, 45, 50], [60, 60], 2),
    ([60, 34, 57, 45, 50], [60] * 3, 3),
    ([60, 34, 57, 45, 50, 40], [60] * 5, 4),
])
def test_fused_roles_in_every_shape(q_bits, p_bits, alpha):
    g, o = pair(14, q_bits, p_bits, alpha)
    level = len(q_bits) - 1
    x = inputs.random_ciphertext_limbs(41, o.primes(), level, o.N)
    ga, oa = g.ct_import(x, level, o.scale), o.ct_import(x, level, o.scale)
    want = [c.limbs() for c in (o.mul(oa, oa), o.mul_relin(oa, oa), o.rescale(oa), o.rotate(oa, 3))]
    saved = g.ntt_get_roles()
    for role in ("modup", "finish", "inverse"):
        for v in SHAPES:
            g.ntt_set_role_variant(hedap.NTT_ROLES[role], v)
            got = [c.limbs() for c in (g.mul(ga, ga), g.mul_relin(ga, ga), g.rescale(ga), g.rotate(ga, 3))]
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), (role, v)
        g.ntt_set_roles(saved)


@pytest.mark.parametrize("log_n", [10, 11, 12, 13])
@pytest.mark.parametrize("v", SHAPES)
def test_small_rings_around_the_cluster_limit(log_n, v):
    """Batches on both sides of 2^21 words; every limb equals that of a batch of its own, a sample the oracle's."""
    import torch
    g, o = pair(log_n, [33, 55, 57, 60], [60], 1)
    primes = o.primes()
    n_l = len(primes)
    most = (1 << 21 >> log_n) // n_l
    g.ntt_set_variant(v, v)
    r = torch.Generator(device="cuda")
    r.manual_seed(log_n)
    for polys, launches in ((most, 1), (most + 1, 2), (2 * most + 3, 2)):
        x = torch.stack([torch.randint(0, int(q), (polys, g.N), generator=r, device="cuda") for q in primes], dim=1)
        x[-1] = torch.tensor([[int(q) - 1] for q in primes], device="cuda")
        for inverse in (False, True):
            n = hedap.launch_count()
            y = g.ntt_batch(x.clone(), n_l, 0, inverse=inverse)
            assert hedap.launch_count() - n == launches
            few = torch.cat([g.ntt_batch(x[k:k + 16].clone(), n_l, 0, inverse=inverse) for k in range(0, polys, 16)])
            assert torch.equal(y, few)
            for k in (0, polys // 2, polys - 1):
                h, hy = x[k].cpu().numpy().view(np.uint64), y[k].cpu().numpy().view(np.uint64)
                for i in range(n_l):
                    assert np.array_equal(hy[i], o.ntt(h[i], i, inverse=inverse)), (polys, inverse, k, i)


@pytest.mark.parametrize("log_n,batch,n_p,alpha", [
    (10, 13, 1, 1), (10, 14, 1, 1), (10, 12, 3, 3), (10, 13, 3, 3), (11, 6, 2, 2), (11, 7, 2, 2), (12, 3, 3, 3), (12, 4, 3, 3)])
def test_products_around_the_separate_inner_product(log_n, batch, n_p, alpha):
    """Q primes of 33 to 60 bits; a digit has just below or just above 2^18 words over the batch."""
    q_bits = [60, 34, 57, 45, 55, 60, 40, 56, 50, 33, 58, 42, 54, 48, 36, 59, 44, 52]
    g, o = pair(log_n, q_bits, [60] * n_p, alpha)
    level = len(q_bits) - 1
    xs = [inputs.random_ciphertext_limbs(70 + k, o.primes(), level, o.N) for k in range(batch)]
    b = g.pack([g.ct_import(x, level, o.scale) for x in xs])
    got, rot = g.mul(b, b), g.rotate(b, 3)
    for k in sorted({0, batch // 2, batch - 1}):
        oa = o.ct_import(xs[k], level, o.scale)
        assert np.array_equal(g.unpack(got, k).limbs(), o.mul(oa, oa).limbs()), k
        assert np.array_equal(g.unpack(rot, k).limbs(), o.rotate(oa, 3).limbs()), k


@pytest.mark.parametrize("log_n", [12, 13])
@pytest.mark.parametrize("n_p,alpha", [(2, 2), (3, 3)])
def test_full_batches_of_small_rings(log_n, n_p, alpha):
    """16 ciphertexts: the fused transforms pass 2^21 words and take the launch shapes; their members alone run as clusters."""
    q_bits = [60, 34, 57, 45, 55, 60, 40, 56, 50, 33] + ([58, 42, 54, 48, 36, 59, 44, 52] if log_n == 12 else [])
    g, o = pair(log_n, q_bits, [60] * n_p, alpha)
    level = len(q_bits) - 1
    xs = [inputs.random_ciphertext_limbs(90 + k, o.primes(), level, o.N) for k in range(16)]
    cts = [g.ct_import(x, level, g.scale) for x in xs]
    b = g.pack(cts)
    for op in (lambda c: g.mul(c, c), lambda c: g.mul_relin(c, c), g.rescale, lambda c: g.rotate(c, 3)):
        got = op(b)
        for k, c in enumerate(cts):
            assert np.array_equal(g.unpack(got, k).limbs(), op(c).limbs()), k
    oa = o.ct_import(xs[5], level, o.scale)
    assert np.array_equal(g.mul(cts[5], cts[5]).limbs(), o.mul(oa, oa).limbs())
