"""Rotations and diagonal products that share one launch: counts beyond a launch's capacity, against the oracle and against
single calls, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu


def pair():
    p = inputs.PRESETS["n10"]
    args = (p["log_n"], p["q_bits"], p["p_bits"], p["alpha"], p["log_scale"], p["hw"], 1)
    return hedap.Context(*args), oracle.Context(*args)


@pytest.mark.parametrize("level", [0, 3, 5])
def test_hoisted_rotations_past_one_launch(level):
    g, o = pair()
    x = inputs.random_ciphertext_limbs(4, o.primes(), level, o.N)
    ga, oa = g.ct_import(x, level, o.scale), o.ct_import(x, level, o.scale)
    steps = list(range(-1, 16)) + [o.N // 2]  # 18 rotations, among them the identity twice
    for s, a, b in zip(steps, g.rotate_hoisted(ga, steps), o.rotate_hoisted(oa, steps)):
        assert np.array_equal(a.limbs(), b.limbs()), s


def test_hoisted_rotations_of_a_batch():
    g, _ = pair()
    cts = [g.ct_import(inputs.random_ciphertext_limbs(30 + k, g.primes(), 4, g.N), 4, g.scale) for k in range(5)]
    steps = [1, 2, 7]
    rot = g.rotate_hoisted(g.pack(cts), steps)
    for k, c in enumerate(cts):
        for a, b in zip(rot, g.rotate_hoisted(c, steps)):
            assert np.array_equal(g.unpack(a, k).limbs(), b.limbs()), k


@pytest.mark.parametrize("log_n,n_q,n_p,alpha,batch,count", [
    (13, 8, 2, 2, 3, 5),   # more than 2^21 words: column and row launches over the parts of all rotations
    (13, 8, 2, 2, 1, 17),  # 16 rotations at once and one by itself
    (10, 10, 8, 8, 2, 3),  # the most special primes a chain may have
])
def test_hoisted_moddown_of_several_rotations(log_n, n_q, n_p, alpha, batch, count):
    """Every rotation of a batch against the oracle's rotations of its members."""
    args = (log_n, [50] * n_q, [60] * n_p, alpha, 50, 64, 1)
    g, o = hedap.Context(*args), oracle.Context(*args)
    level = n_q - 1
    x = [inputs.random_ciphertext_limbs(50 + k, o.primes(), level, o.N) for k in range(batch)]
    steps = [k - 1 for k in range(count)]
    rot = g.rotate_hoisted(g.pack([g.ct_import(v, level, o.scale) for v in x]), steps)
    for k, v in enumerate(x):
        for a, b in zip(rot, o.rotate_hoisted(o.ct_import(v, level, o.scale), steps)):
            assert np.array_equal(g.unpack(a, k).limbs(), b.limbs()), k


@pytest.mark.parametrize("inverse", [True, False])
def test_diagonal_products_past_one_launch(inverse):
    """One grouped factor over all 512 slots: 64 giant steps of 16 baby steps."""
    g, o = pair()
    bts = dict(K=28, r=0, deg=2, cts=1, stc=1)
    assert g.bts_setup(**bts) == o.bts_setup(**bts)
    z = inputs.uniform_values(7, o.N // 2, -1, 1)
    oc = o.encrypt(z, o.n_q - 1, 9)
    gc = g.ct_import(oc.limbs(), oc.level, oc.scale)
    a = g.linear_transform_group(gc, 1, inverse, 0, oc.scale / 16)
    b = o.linear_transform_group(oc, 1, inverse, 0, oc.scale / 16)
    assert a.level == b.level and np.array_equal(a.limbs(), b.limbs())
