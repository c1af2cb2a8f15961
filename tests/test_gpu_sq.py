"""S(q) on the GPU against the oracle at the edges of the kernel's split (rows
per warp, 32-column blocks, planes, several bins per block, unequal spacings):
bin counts exactly, sums to FP64 rounding."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2405_02410_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nbins", [1, 7, 64, 500])
@pytest.mark.parametrize("shape,dx", [((4,), (1.0,)), ((1024,), (0.3,)), ((4, 4), (1.0, 1.0)), ((64, 64), (1.0, 1.0)),
                                      ((512, 128), (0.5, 2.0)), ((128, 1024), (1.0, 0.7)), ((1024, 512), (1.0, 1.0)),
                                      ((8, 4, 16), (1.0, 1.0, 1.0)), ((64, 32, 64), (1.0, 0.5, 2.0))])
def test_matches_oracle(shape, dx, nbins, prec):
    from paper_2405_02410_gb300 import pss
    s = pss.System(shape, dt=0.1, precision=prec, dx=dx)
    f = s.add_field("phi")
    x = np.random.default_rng(5).standard_normal(shape)
    s.set_field(f, x)
    full = np.fft.fftn(np.fft.irfftn(s.get_spectrum(f).astype(np.complex128), s=shape, axes=tuple(range(len(shape)))))
    m = O.Model(shape=shape, dt=0.1, dx=tuple(dx) + (1.0,) * (3 - len(dx)))
    S0, cnt0, L0 = O.structure_factor(m, full, nbins)
    S, cnt, L = s.structure_factor(f, nbins)
    np.testing.assert_array_equal(cnt, cnt0)
    # sums of at most 2^19 positive terms, each a few roundings
    np.testing.assert_allclose(S, S0, rtol=1e-11, atol=0)
    assert abs(L - L0) <= 1e-11 * max(abs(L0), 1e-300)
