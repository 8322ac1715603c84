"""The tail's noise transform, two samples at a time with its own quotients: bit for bit the
oracle's over enough words to meet most of the 2^23 uniforms, across ragged ends."""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,rir,k0,n", [(1, 0, 0, 1 << 24), (2 ** 63 + 5, 77, 3, 100001), (9, 5, 2, 1)])
def test_bits(seed, rir, k0, n):
    import __graft_entry__
    __graft_entry__.build()
    z = ism.ism_diffuse_noise(seed, rir, k0, n).cpu().numpy()
    assert np.array_equal(z.view(np.uint32), oracle.noise(seed, rir, k0, n).view(np.uint32))
