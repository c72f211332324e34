"""Transforms that multiply by halves (N >= 8192, primes below 2^55) against the
CPU reference, at the sizes where their tiling can go wrong: the fewest and
ragged counts of polynomials per limb, the smallest column and chunk lengths,
the widest primes that take this form and the first that do not, and the inputs
that grow the lazy words most. Exact integer arithmetic: the tolerance is zero."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

RING = {"2N": 0, "3N": 3, "5N/2": 5}


def pair(ring, logN, bits, L, alpha=1, keys=False):
    import paper_2604_19890_gb300 as ssg
    kw = dict(logN=logN, L=L, alpha=alpha, bits=bits, p=17, r=1, h=8, seed=23, m_odd=RING[ring])
    g, o = ssg.Context(nmax=0, **kw), O.Oracle(**kw)
    if keys:
        g.keygen([])
        o.keygen([])
    return g, o


@pytest.mark.parametrize("outer", [1, 2, 3, 5, 9])
@pytest.mark.parametrize("ring,logN,bits", [("2N", 13, 55), ("2N", 14, 36), ("2N", 15, 55), ("2N", 13, 56),
                                            ("3N", 13, 55), ("3N", 14, 55), ("5N/2", 13, 55), ("5N/2", 14, 36)])
def test_transform_counts_and_extremes(ring, logN, bits, outer):
    import torch
    L = 2
    g, o = pair(ring, logN, bits, L)
    rng = np.random.default_rng(100 * logN + outer)
    data = np.stack([rng.integers(0, int(g.primes[i % L]), g.N, dtype=np.uint64) for i in range(outer * L)])
    for i in range(L):  # the first polynomials: every word q - 1; q - 1 in the upper half, in every other word
        q = int(g.primes[i])
        data[i] = q - 1
        if outer > 1:
            data[L + i] = 0
            data[L + i, g.N // 2:] = q - 1
        if outer > 2:
            data[2 * L + i] = 0
            data[2 * L + i, ::2] = q - 1
    t = torch.from_numpy(data.view(np.int64).copy()).cuda()
    g.ntt_forward(t, 0, L)
    fw = t.cpu().numpy().view(np.uint64).copy()
    for j in range(min(outer * L, 6)):
        assert (fw[j] == o.ntt_fwd(j % L, data[j])).all(), j
    assert (fw[-1] == o.ntt_fwd(L - 1, data[-1])).all()
    g.ntt_inverse(t, 0, L)
    assert (t.cpu().numpy().view(np.uint64) == data).all()
    t = torch.from_numpy(data.view(np.int64).copy()).cuda()  # the same words as values: the inverse's own extremes
    g.ntt_inverse(t, 0, L)
    inv = t.cpu().numpy().view(np.uint64)
    for j in range(min(outer * L, 6)):
        assert (inv[j] == o.ntt_inv(j % L, data[j])).all(), j


@pytest.mark.parametrize("count,level", [(1, 2), (3, 5), (5, 4)])
@pytest.mark.parametrize("ring,bits", [("2N", 55), ("3N", 36), ("5N/2", 55), ("2N", 57)])
def test_multiplication_with_ragged_digits(ring, bits, count, level):
    """Groups of polynomials that leave out a digit's own limbs (the last digit shorter than alpha)."""
    g, o = pair(ring, 13, bits, 5, alpha=2, keys=True)
    rng = np.random.default_rng(count)
    vals = rng.integers(0, g.t, (2, count, g.slots))
    a, b = (g.encrypt(np.stack([g.encode(v) for v in vals[k]]), 10 + 20 * k) for k in (0, 1))
    oa, ob = ([o.encrypt(o.encode(v), 10 + 20 * k + i) for i, v in enumerate(vals[k])] for k in (0, 1))
    if level < 5:
        a, b = g.modswitch(a, 5 - level), g.modswitch(b, 5 - level)
        oa, ob = [o.modswitch(x, 5 - level) for x in oa], [o.modswitch(x, 5 - level) for x in ob]
    w = g.mul_relin(a, b).words()
    for i in (0, count - 1):
        assert (w[i] == o.mul(oa[i], ob[i]).words()).all()


@pytest.mark.parametrize("level", [14, 15, 16, 17])
@pytest.mark.parametrize("count", [1, 2])
def test_digit_counts_around_the_fused_limit(count, level):
    """Key switches of one-prime digits where the fused inner product's rows fill a CTA (15 digits and the
    correction's two less one) and where they no longer fit, through a relinearisation and a multiplication."""
    import paper_2604_19890_gb300 as ssg
    kw = dict(logN=13, L=17, alpha=1, bits=50, p=17, r=1, h=8, seed=29, m_odd=0)
    g, o = ssg.Context(nmax=0, **kw), O.Oracle(**kw)
    g.keygen([])
    o.keygen([])
    rng = np.random.default_rng(level)
    vals = rng.integers(0, g.t, (count, g.slots))
    a = g.encrypt(np.stack([g.encode(v) for v in vals]), 3)
    oa = [o.encrypt(o.encode(v), 3 + i) for i, v in enumerate(vals)]
    if level < 17:
        a, oa = g.modswitch(a, 17 - level), [o.modswitch(x, 17 - level) for x in oa]
    rel, mul = g.relin(g.mul(a, a)).words(), g.mul_relin(a, a).words()
    assert (rel[-1] == o.relin(o.tensor(oa[-1], oa[-1])).words()).all()
    assert (mul[0] == o.mul(oa[0], oa[0]).words()).all()


@pytest.mark.parametrize("nin,nout", [(1, 1), (2, 16), (7, 3), (15, 8), (16, 16)])
@pytest.mark.parametrize("bits,logN", [(36, 9), (55, 13), (58, 8)])
def test_small_coefficient_combinations(bits, logN, nin, nout):
    """sum_i c_i y_i with |c_i| < 2^27: the largest sums of each sign, words q - 1, zeros, and rows one past the bound."""
    import paper_2604_19890_gb300 as ssg
    g = ssg.Context(logN=logN, L=3, alpha=1, bits=bits, p=17, r=1, h=8, seed=5, nmax=0)
    rng = np.random.default_rng(nin)
    level, top = 2, (1 << 27) - 1
    w = np.stack([np.stack([rng.integers(0, int(g.primes[i]), (1, 2, g.N), dtype=np.uint64) for i in range(level)], 2)
                  for _ in range(nin)])  # [nin][1][2][level][N]
    for i in range(level):
        w[:, 0, 0, i, ::3] = int(g.primes[i]) - 1
        w[:, 0, 1, i, ::5] = 0
    rows = rng.integers(-top, top + 1, (nout, nin))
    rows[0] = top
    rows[-1] = -top
    if nout > 2:
        rows[1, 0] = 0
        rows[2, -1] = top + 1 if nin == 7 else top  # 2^27 takes the wider path for the whole call
    outs = g.linear_combinations([g.from_words(x, 1) for x in w], rows.tolist())
    for j in (0, nout - 1, nout // 2):
        got = outs[j].words()[0]
        for i in range(level):
            q = int(g.primes[i])
            exp = sum(int(rows[j, t]) * w[t, 0, :, i, :].astype(object) for t in range(nin)) % q
            assert (got[:, i, :].astype(object) == exp).all(), (j, i)


@pytest.mark.parametrize("logN", [9, 13])
def test_arrays_between_16_byte_boundaries(logN):
    """The raw transform, the encryption and the multiplication take outputs that start on any word."""
    import ctypes as C

    import torch

    import paper_2604_19890_gb300 as ssg
    g = ssg.Context(logN=logN, L=3, alpha=2, bits=50, p=17, r=1, h=8, seed=31, nmax=0)
    g.keygen([])
    rng = np.random.default_rng(logN)
    data = np.stack([rng.integers(0, int(g.primes[i % 3]), g.N, dtype=np.uint64) for i in range(6)])
    even = torch.from_numpy(data.view(np.int64).copy()).cuda()
    odd = torch.zeros(6 * g.N + 1, dtype=torch.int64, device="cuda")[1:]
    odd.copy_(even.flatten())
    assert odd.data_ptr() % 16 == 8
    for f in (g.ntt_forward, g.ntt_inverse):
        f(even, 0, 3)
        f(odd, 0, 3)
        assert torch.equal(odd, even.flatten())
    m = np.stack([g.encode(rng.integers(0, g.t, g.slots)) for _ in range(2)])
    a = g.encrypt(m, 5)
    flat = torch.zeros(a.buf.numel() + 1, dtype=torch.int64, device="cuda")[1:]
    d = a.desc()
    d.data = flat.data_ptr()
    dm = torch.from_numpy(m.view(np.int64).copy()).cuda()
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert ssg.lib().ss_encrypt(g.h, C.c_void_p(dm.data_ptr()), 2, 5, a.t_exp, C.byref(d), st) == ssg.SS_OK
    assert torch.equal(flat, a.buf.flatten())
    p = g.mul_relin(a, a)
    flat = torch.zeros(p.buf.numel() + 1, dtype=torch.int64, device="cuda")[1:]
    da, do = a.desc(), p.desc()
    do.data = flat.data_ptr()
    assert ssg.lib().ss_mul_relin(g.h, C.byref(da), C.byref(da), C.byref(do), st) == ssg.SS_OK
    assert torch.equal(flat, p.buf.flatten()) and (do.level, do.ncomp) == (p.level, p.ncomp)
