"""The row kernel that evaluates all product terms of an FP32 instance
(k_row_terms) against the factor-by-factor launches, over the forms its rule
accepts, and the forms it leaves to them.

Bar: rel-L2 <= 1e-5 (FP32 rounding of two evaluation orders over a few steps)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2405_02410_gb300 import build
    build.build()


def pss():
    from paper_2405_02410_gb300 import pss as m
    return m


def _lhs(s, f):
    s.add_term(f, True, [(-1, 0.5, 0), (-1, 0.7, 1), (-1, 0.3, 2)], [(f, 1)])


def coupled(s):     # two operators on one field, multiples of q^2
    f, g = s.add_field("f"), s.add_field("g")
    b, c, d = s.add_param("b", 1.0), s.add_param("c", 0.5), s.add_param("D", 0.05)
    for x in (f, g):
        _lhs(s, x)
    s.add_term(f, False, [(b, -1.0, 1)], [(f, 3)])
    s.add_product_term(f, [(c, -1.0, 1), (b, -0.25, 1)], [(f, 1), (g, 2)])
    s.add_product_term(g, [(-1, -0.7, 0), (-1, 0.1, 1)], [(f, 2), (g, 1)])
    s.set_noise(f, d, 1)
    s.set_noise(g, d, 0)
    return 2, True


def burgers(s):     # x and y derivatives, a Laplacian, a field squared, a plain power field beside
    h, k = s.add_field("h"), s.add_field("k")
    d = s.add_param("D", 0.05)
    for x in (h, k):
        _lhs(s, x)
    s.add_product_term(h, [(-1, 0.3, 0)], [(h, 1), (h, 1, 0, 0)])
    if s.dim == 2:
        s.add_product_term(h, [(-1, 0.3, 0)], [(h, 2, 1, 0)])
    s.add_product_term(h, [(-1, 0.02, 0)], [(k, 1, -1, 1), (h, 1)])
    s.add_term(k, False, [(-1, -0.8, 1)], [(k, 3)])
    s.set_dealias(k, 3)
    s.set_noise(h, d, 0)
    return 2, True


def kpz(s):
    pss().add_kpz_field(s, sigma=1.0, lam=0.6, D=0.02, dealias_order=0)
    return 1, True


def three_targets(s):   # every field of four a factor
    fs = [s.add_field(f"f{i}") for i in range(4)]
    for f in fs:
        _lhs(s, f)
    s.add_product_term(fs[0], [(-1, 0.2, 1)], [(fs[1], 1), (fs[2], 1), (fs[3], 2)])
    s.add_product_term(fs[1], [(-1, 0.2, 0)], [(fs[0], 4)])
    s.add_product_term(fs[2], [(-1, 0.2, 0)], [(fs[0], 1), (fs[1], 1)])
    return 4, True


def two_operators(s):   # operators of different powers: factor by factor
    f = s.add_field("f")
    _lhs(s, f)
    s.add_product_term(f, [(-1, 0.2, 1)], [(f, 2)])
    s.add_product_term(f, [(-1, 0.2, 0)], [(f, 3)])
    return 1, False


def _system(shape, form, fuse, batch=1, prec="f32", frame=False):
    s = pss().System(shape, dt=0.01, seed=3, batch=batch, precision=prec, dx=(1.0, 0.8, 1.0))
    nf, fused = form(s)
    s.set_tuning("fuse_terms", fuse)
    s.set_tuning("resident", 0)
    s.set_tuning("persist", 0)
    if frame:
        s.set_frame(0, 3, 0.2, -0.1)
    for b in range(batch):
        s.select_instance(b)
        for f in range(nf):
            s.init_uniform(f, -0.4, 0.4)
    return s, nf, fused


def _spectra(s, nf):
    out = []
    for b in range(s.batch):
        s.select_instance(b)
        out += [s.get_spectrum(f) for f in range(nf)]
    return out


def _agree(a, b):
    for x, y in zip(a, b):
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y), np.linalg.norm(x - y) / np.linalg.norm(y)


@pytest.mark.parametrize("batch,frame", [(1, False), (3, False), (2, True)])
@pytest.mark.parametrize("form", [coupled, burgers, kpz, three_targets, two_operators])
@pytest.mark.parametrize("shape", [(4, 4), (64, 64), (256, 256), (8, 1024), (1024, 16), (128,), (16,)])
def test_agrees_with_the_launches_per_factor(shape, form, batch, frame):
    if frame and shape[-1] < 8:
        pytest.skip("the frame does not fit")
    a, nf, fused = _system(shape, form, 1, batch, frame=frame)
    b, _, _ = _system(shape, form, 0, batch, frame=frame)
    la = a.launch_count
    a.step(1)
    la, lb = a.launch_count - la, b.launch_count
    b.step(1)
    lb = b.launch_count - lb
    assert la < lb if fused else la == lb
    a.step(6)
    b.step(6)
    _agree(_spectra(a, nf), _spectra(b, nf))
    assert a.get_step() == b.get_step() == 7


def test_parameters_terms_and_switches_mid_run():
    shape = (64, 32)
    a, nf, _ = _system(shape, coupled, 1, 2)
    b, _, _ = _system(shape, coupled, 0, 2)
    for s in (a, b):
        s.step(3)
        s.set_param_batch(1, np.array([0.2, 0.9]))
        s.step(3)
        s.add_term(1, False, [(-1, -0.5, 0), (-1, 0.1, 1)], [(1, 2)])
        s.step(3)
    a.set_tuning("fuse_terms", 0)
    a.step(2)
    a.set_tuning("fuse_terms", 1)
    a.step(2)
    b.step(4)
    _agree(_spectra(a, nf), _spectra(b, nf))


def test_fp64_keeps_the_launches_per_factor():
    a, nf, _ = _system((32, 32), coupled, 1, prec="f64")
    b, _, _ = _system((32, 32), coupled, 0, prec="f64")
    la, lb = a.launch_count, b.launch_count
    a.step(4)
    b.step(4)
    assert a.launch_count - la == b.launch_count - lb
    for x, y in zip(_spectra(a, nf), _spectra(b, nf)):
        assert x.tobytes() == y.tobytes()
