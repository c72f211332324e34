"""Merged lanes of the batched form (ss_batch_config with nstreams = 0) on rings N >= 8192, for primes on
both sides of the width up to which transforms multiply by halves and are merged: launches of the lanes, and
words equal to the CPU reference, alone and beside lanes of the other width."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

RING = {"2N": 0, "3N": 3, "5N/2": 5}


def pair(ring, logN, bits):
    import paper_2604_19890_gb300 as ssg
    kw = dict(logN=logN, L=4, alpha=2, bits=bits, p=17, r=1, h=8, seed=bits, m_odd=RING[ring])
    g, o = ssg.Context(nmax=0, **kw), O.Oracle(**kw)
    g.keygen([])
    o.keygen([])
    return g, o


def products(world, items, seed):
    """Pairs of fresh ciphertexts of contexts `items`, and their products by the CPU reference."""
    rng = np.random.default_rng(seed)
    pairs, refs = [], []
    for i, ci in enumerate(items):
        g, o = world[ci]
        v = rng.integers(0, g.t, (2, g.slots))
        pairs.append((ci, *(g.encrypt(g.encode(v[k]), 10 + 2 * i + k) for k in (0, 1)), False))
        refs.append(o.mul(*(o.encrypt(o.encode(v[k]), 10 + 2 * i + k) for k in (0, 1))).words())
    return pairs, refs


def launches_of(world, pairs):
    """Launches of one run with one lane per pair, and the products' words."""
    import torch

    import paper_2604_19890_gb300 as ssg
    gs = [g for g, _ in world]
    b = ssg.Batch(gs, pairs)
    b.config(1, 0)
    st = torch.cuda.Stream()
    n0 = sum(g.launches() for g in gs)
    b.run(st)
    st.synchronize()
    n = sum(g.launches() for g in gs) - n0
    words = [p.words()[0] for p, _ in b.results()]
    b.close()
    return n, words


@pytest.mark.parametrize("ring,logN,bits", [("2N", 13, 55), ("2N", 13, 56), ("3N", 14, 58), ("5N/2", 13, 56),
                                            ("5N/2", 14, 57)])
def test_lanes_share_transforms_by_halves_and_inner_products(ring, logN, bits):
    world = [pair(ring, logN, bits)]
    pairs, refs = products(world, [0, 0, 0], bits)
    one, w1 = launches_of(world, pairs[:1])
    three, w3 = launches_of(world, pairs)
    assert all((w == r).all() for w, r in zip(w1 + w3, refs[:1] + refs))
    # a product has two inner products, launched once for all lanes, and four transforms of two launches each, which
    # the lanes share where they multiply by halves
    assert three == one + 2 * (one - (10 if bits <= 55 else 2))


def test_lanes_of_both_widths_beside_each_other():
    world = [pair("2N", 13, 55), pair("3N", 13, 57), pair("2N", 14, 58), pair("5N/2", 13, 36)]
    pairs, refs = products(world, [0, 1, 2, 3, 1], 7)
    _, words = launches_of(world, pairs)
    assert all((w == r).all() for w, r in zip(words, refs))


@pytest.mark.parametrize("bits,tiles", [(55, 1), (56, 2)])
def test_the_tuner_runs_each_different_setting_twice(bits, tiles):
    """The transform's tile is a choice on primes of more than 55 bits only; elsewhere the tuner leaves it as it was."""
    import torch

    import paper_2604_19890_gb300 as ssg
    world = [pair("2N", 13, bits)]
    pairs, _ = products(world, [0] * 9, bits)
    g = world[0][0]
    b = ssg.Batch([g], pairs)
    st = torch.cuda.Stream()
    n = 0
    for chunk in (8, 32, 64):
        for streams in (1, 3, 0):
            b.config(chunk, streams)
            n0 = g.launches()
            b.run(st)
            st.synchronize()
            n += g.launches() - n0
    b.config(8, 1, 12)
    n0 = g.launches()
    best = b.tune(st)
    assert g.launches() - n0 == 2 * tiles * n
    assert best[2] == 12 or tiles > 1
    b.close()
