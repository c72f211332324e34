"""Device scratch of single calls: a call that is refused gives back what it took from the
stream-ordered pool, and a transform in place takes nothing where its kernels read single words."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, CU_MEMPOOL_ATTR_USED_MEM_HIGH


class Pool:
    """Bytes in use of the current device's default memory pool (driver API: one pool per device and process)."""

    def __init__(self):
        import torch
        self.torch = torch
        torch.zeros(1, device="cuda")
        self.cu = C.CDLL("libcuda.so.1")
        dev, self.pool = C.c_int(), C.c_void_p()
        assert self.cu.cuDeviceGet(C.byref(dev), torch.cuda.current_device()) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(C.byref(self.pool), dev) == 0

    def get(self, attr=USED_CURRENT):
        self.torch.cuda.synchronize()
        v = C.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, C.byref(v)) == 0
        return v.value

    def reset_high(self):
        v = C.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_HIGH, C.byref(v)) == 0


def context(**kw):
    import paper_2604_19890_gb300 as ssg
    return ssg.Context(alpha=1, p=17, r=1, h=4, seed=37, nmax=0, **kw)


# more than 65535 polynomials in one transform are refused
def test_refused_calls_give_back_their_scratch():
    import paper_2604_19890_gb300 as ssg
    g = context(logN=4, L=2, bits=36)
    g.keygen([])
    pool = Pool()
    x = g.from_words(np.zeros((32768, 2, 2, g.N), dtype=np.uint64), 1)
    before = pool.get()
    with pytest.raises(ssg.SSError):
        g.encrypt(np.zeros((32769, g.N), dtype=np.uint64), 1)
    assert pool.get() == before
    with pytest.raises(ssg.SSError):
        g.modswitch(x, 1)
    assert pool.get() == before


def test_refused_raw_transform_gives_back_its_scratch():
    import torch

    import paper_2604_19890_gb300 as ssg
    g = context(logN=13, L=1, bits=36)
    pool = Pool()
    odd = torch.zeros(65536 * g.N + 1, dtype=torch.int64, device="cuda")[1:].view(65536, g.N)
    assert odd.data_ptr() % 16 == 8
    before = pool.get()
    for f in (g.ntt_forward, g.ntt_inverse):
        with pytest.raises(ssg.SSError):
            f(odd, 0, 1)
        assert pool.get() == before


# single-phase transforms and the form of wide primes read words one by one, so any start of an array will do
@pytest.mark.parametrize("logN,bits", [(9, 55), (13, 56)])
def test_transform_between_16_byte_boundaries_stays_in_place(logN, bits):
    import torch
    g = context(logN=logN, L=2, bits=bits)
    pool = Pool()
    even = torch.stack([torch.arange(g.N, device="cuda") * (i + 7) for i in range(4)])
    odd = torch.zeros(even.numel() + 1, dtype=torch.int64, device="cuda")[1:].view_as(even)
    odd.copy_(even)
    assert odd.data_ptr() % 16 == 8
    for f in (g.ntt_forward, g.ntt_inverse):
        f(even, 0, 2)
        before = pool.get()
        pool.reset_high()
        f(odd, 0, 2)
        assert pool.get(USED_HIGH) <= before
        assert torch.equal(odd, even)
