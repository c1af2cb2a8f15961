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


@pytest.mark.parametrize("shape,nbins", [((640, 480), 64), ((640, 480), 16), ((100, 100), 49), ((63, 77), 49),
                                         ((128, 64), 64), ((45,), 16), ((12, 20, 28), 32)])
def test_torch_bins_of_any_shape(shape, nbins):
    # a mode on a bin's edge belongs to the bin below: ceil(|q| nbins dx / pi) - 1 with every
    # operation correctly rounded, as numpy's are; bin counts and sums of |phi|^2 = 1
    import torch
    from paper_2405_02410_gb300 import autograd as A
    h = torch.ones(shape[:-1] + (shape[-1] // 2 + 1,), dtype=torch.complex128, device="cuda")
    S, cnt = A.binned_structure_factor(h, shape, nbins)
    ks = [np.rint(np.fft.fftfreq(m) * m) for m in shape[:-1]] + [np.arange(shape[-1] // 2 + 1)]
    g = np.meshgrid(*ks, indexing="ij")
    s2 = sum((2.0 * nbins * k / m) ** 2 for k, m in zip(g, shape))
    s = np.sqrt(s2)
    valid = (s2 > 0) & (s <= nbins)
    w = np.where((g[-1] == 0) | (2 * g[-1] == shape[-1]), 1.0, 2.0) * valid
    want = np.bincount(np.where(valid, np.ceil(s) - 1, 0).astype(int).reshape(-1), w.reshape(-1), minlength=nbins)
    np.testing.assert_array_equal(cnt.cpu().numpy(), want)
    np.testing.assert_allclose(S.cpu().numpy(), np.where(want > 0, 1.0 / np.prod(shape), 0.0), rtol=1e-12)
