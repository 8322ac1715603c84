"""The tail's noise transform over every one of the 2^23 uniforms, in both places of the pair that
it takes at a time: bit for bit the oracle's.  The words are Philox4x32-10's own, 32 of them to a
uniform and place (all are met: counted)."""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N_UNIFORMS = 1 << 23
CHUNK = 1 << 26   # samples a call


def _words(seed, rir, n):
    """Philox4x32-10, counter (k / 4, rir, 0, 0): the words of samples 0 .. n - 1."""
    m32 = 0xFFFFFFFF

    def mul(m, a):   # high and low words of the 64-bit product, in signed arithmetic
        lo, hi = m * (a & 0xFFFF), m * (a >> 16)
        top = hi + (lo >> 16)
        return top >> 16, ((top & 0xFFFF) << 16) | (lo & 0xFFFF)

    c = [torch.arange(n // 4, device="cuda"), *(torch.full((n // 4,), v, dtype=torch.int64, device="cuda") for v in (rir, 0, 0))]
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return torch.stack(c, 1)


def test_every_uniform_in_both_places():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    f = oracle._load().oracle_logistic_f32
    table = np.fromiter(map(f, ((np.arange(N_UNIFORMS) + 0.5) * 2.0 ** -23).tolist()), np.float32, N_UNIFORMS)
    table = torch.from_numpy(table.view(np.int32)).cuda()
    met = torch.zeros((2, N_UNIFORMS), dtype=torch.bool, device="cuda")
    for rir in range(8):
        z = ism.ism_diffuse_noise(11, rir, 0, CHUNK).view(torch.int32).reshape(-1, 4)
        u = _words(11, rir, CHUNK) >> 9
        assert torch.equal(z, table[u])
        for place in (0, 1):
            met[place, u[:, place::2].reshape(-1)] = True
    assert bool(met.all())
