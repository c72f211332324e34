"""The two tile sizes of the transforms' column phase on both sides of the count of polynomials at which the
larger one takes over (two waves of four 4096-word tiles an SM): first, middle and last polynomials against the
CPU reference, all of them against the same transform in small groups. Exact: the tolerance is zero."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

RING = {"2N": 0, "3N": 3, "5N/2": 5}


@pytest.mark.parametrize("ring,logN,bits", [("2N", 13, 55), ("2N", 14, 55), ("2N", 15, 36), ("2N", 16, 55),
                                            ("3N", 13, 36), ("3N", 14, 55), ("3N", 15, 55), ("3N", 16, 36),
                                            ("5N/2", 13, 55), ("5N/2", 14, 36), ("5N/2", 15, 55), ("5N/2", 16, 55)])
def test_column_tiles_around_their_limit(ring, logN, bits):
    import torch

    import paper_2604_19890_gb300 as ssg
    kw = dict(logN=logN, L=1, alpha=1, bits=bits, p=17, r=1, h=8, seed=23, m_odd=RING[ring])
    g, o = ssg.Context(nmax=0, **kw), O.Oracle(**kw)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    least = -(-(8 * sms) // (1 << (logN - 12)))  # polynomials from which the larger tile runs
    q = int(g.primes[0])
    gen = torch.Generator(device="cuda").manual_seed(logN)
    for count in (least - 1, least, least + 1):
        data = torch.randint(0, q, (count, g.N), generator=gen, dtype=torch.int64, device="cuda")
        data[0] = q - 1  # the words that grow the lazy sums most
        data[count // 2] = 0
        data[count // 2, g.N // 2:] = q - 1
        data[-1] = 0
        data[-1, ::2] = q - 1
        host = {j: data[j].cpu().numpy().view(np.uint64) for j in (0, 1, count // 2, count - 1)}
        for f, ref in ((g.ntt_forward, o.ntt_fwd), (g.ntt_inverse, o.ntt_inv)):
            whole, parts = data.clone(), data.clone()
            f(whole, 0, 1)
            for i in range(0, count, 16):
                f(parts[i:i + 16], 0, 1)
            assert torch.equal(whole, parts)
            for j, x in host.items():
                assert (whole[j].cpu().numpy().view(np.uint64) == ref(0, x)).all(), (count, j)
