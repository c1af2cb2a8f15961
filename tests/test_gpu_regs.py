"""The register passes of FP32 2D and 3D systems (tuning key "regs") against
the staged kernels over the sides, orders, operators and batches the rule that
selects them accepts (and sides where only some of the passes are taken),
and against the oracle.

Bars: rel-L2 <= 1e-5 against the staged kernels (FP32 rounding of two transform
orders over a few steps, as for the 2D paths); rel-L2 <= 1e-4 per mode against
the FP64 oracle.
"""
import numpy as np
import pytest

from oracle import oracle as O

from tests.parity import check_spectrum
from tests.test_gpu_terms_fused import _system as _terms_system, burgers, coupled, kpz, three_targets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2405_02410_gb300 import build
    build.build()


def _system(shape, regs, fields=1, batch=1, order=2, noisy=True, power=3):
    from paper_2405_02410_gb300 import pss as P
    s = P.System(shape, dt=0.01, seed=5, batch=batch, precision="f32", dx=(1.0, 0.7, 1.3))
    for i in range(fields):
        f = s.add_field(f"f{i}")
        pa, pD = s.add_param(f"a{i}", -0.8), s.add_param(f"D{i}", 0.05)
        up = i % 2   # non-conserved, then conserved with an operator of degree 3 in q^2
        s.add_term(f, True, [(pa, 1.0, up), (-1, 1.0, 1 + up)] + ([(-1, 0.01, 3)] if up else []), [(f, 1)])
        if power:
            s.add_term(f, False, [(-1, -1.0, up)], [(f, power)])
        if noisy:
            s.set_noise(f, pD, up)
        s.set_dealias(f, order)
    s.set_tuning("regs", regs)
    if len(shape) == 2 and regs != 1:   # the per-step kernels at every size
        s.set_tuning("resident", 0)
        s.set_tuning("persist", 0)
    for b in range(batch):
        s.select_instance(b)
        for f in range(fields):
            s.init_uniform(f, -0.2, 0.2)
    return s


def _results(s, fields):
    out = []
    for b in range(s.batch):
        s.select_instance(b)
        for f in range(fields):
            out += [s.get_spectrum(f), s.get_field(f)]
    return out


@pytest.mark.parametrize("shape,kw", [
    ((16, 16, 16), {}), ((16, 4, 8), dict(fields=2)), ((32, 64, 8), dict(order=3)), ((64, 32, 16), dict(fields=2)),
    ((128, 16, 32), dict(order=0)), ((256, 8, 16), dict(noisy=False)), ((4, 256, 8), {}), ((8, 128, 64), dict(fields=2)),
    ((64, 128, 4), dict(batch=3, fields=2)), ((512, 16, 4), {}), ((16, 512, 4), {}), ((32, 32, 64), dict(power=0)),
    ((16, 32, 128), dict(power=2, order=1)), ((256, 64, 32), dict(fields=2)),
    ((8, 4, 256), dict(order=0)), ((16, 16, 512), {}), ((4, 4, 32), dict(power=1, order=4)), ((4, 8, 16), dict(batch=2)),
    ((16, 64, 256), dict(fields=2)),
])
def test_against_the_staged_kernels(shape, kw):
    fields = kw.get("fields", 1)
    got = []
    for regs in (1, 0):
        s = _system(shape, regs, **kw)
        s.step(1)
        s.step(4)
        got.append(_results(s, fields))
        s.close()
    for x, y in zip(*got):
        assert np.isfinite(x).all()
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)


@pytest.mark.parametrize("shape,kw", [
    ((16, 16), {}), ((32, 64), dict(fields=2)), ((64, 32), dict(order=3)), ((128, 256), dict(order=0)),
    ((256, 128), dict(batch=3, fields=2)), ((512, 16), dict(noisy=False)), ((16, 512), {}), ((512, 512), dict(fields=2)),
    ((1024, 32), {}), ((32, 1024), dict(power=2)), ((1024, 1024), dict(order=0)), ((512, 1024), dict(power=0)),
])
def test_2d_against_the_staged_kernels(shape, kw):
    fields = kw.get("fields", 1)
    got = []
    for regs in (2, 0):
        s = _system(shape, regs, **kw)
        s.step(1)
        s.step(4)
        got.append(_results(s, fields))
        s.close()
    for x, y in zip(*got):
        assert np.isfinite(x).all()
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)


@pytest.mark.parametrize("shape,batch,fields", [((512, 512), 9, 1), ((256, 256), 33, 1), ((512, 1024), 3, 1), ((1024, 1024), 1, 2)])
def test_2d_systems_that_fill_the_chip(shape, batch, fields):
    # by the rule's own choice, each instance against the staged kernels
    s = _system(shape, 1, batch=batch, fields=fields)
    s.step(3)
    got = _results(s, fields)
    s.close()
    r = _system(shape, 0, batch=batch, fields=fields)
    r.step(3)
    for x, y in zip(got, _results(r, fields)):
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)
    r.close()


def test_2d_path_changes_between_runs():
    # the per-step kernels keep the product in another layout than the register passes
    s, r = _system((256, 256), 2), _system((256, 256), 0)
    for regs in (0, 2, 0):
        s.set_tuning("regs", regs)
        s.step(2)
        r.step(2)
    for x, y in zip(_results(s, 1), _results(r, 1)):
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)
    s.close()
    r.close()


@pytest.mark.parametrize("shape", [(16, 32, 16), (64, 16, 8), (128, 4, 16), (8, 64, 32), (16, 16, 256)])
def test_against_the_oracle(shape):
    from paper_2405_02410_gb300 import pss as P
    kw = dict(dt=0.01, a=-1.0, b=1.0, K=1.0, D=0.05, seed=7)
    s = P.model_b(shape, precision="f32", **kw)
    s.init_uniform(0, -0.1, 0.1)
    s.step(10)
    m = O.model_b(shape, **kw)
    ref = O.half(O.run(m, O.to_spectrum(m, O.init_uniform(m, -0.1, 0.1)), 0, 10))
    check_spectrum(s.get_spectrum(0), ref, 1e-4)
    s.close()


def test_a_state_that_is_not_finite_is_reported():
    from paper_2405_02410_gb300 import pss as P
    s = _system((32, 16, 16), 1, noisy=False)
    h = s.get_spectrum(0)
    h[3, 2, 5] = np.inf
    s.set_spectrum(0, h)
    s.step(1)
    with pytest.raises(P.PssError):
        s.get_spectrum(0)
    s.close()


@pytest.mark.parametrize("form", [coupled, burgers, kpz, three_targets])
@pytest.mark.parametrize("shape,batch", [((8, 16), 1), ((16, 32), 2), ((4, 64), 1), ((64, 128), 1), ((32, 256), 3)])
def test_product_terms_against_the_staged_row_kernel(shape, batch, form):
    got = []
    for regs in (1, 0):
        s, nf, _ = _terms_system(shape, form, 1, batch)
        s.set_tuning("regs", regs)
        s.step(3)
        got.append(_results(s, nf))
        assert s.get_step() == 3
        s.close()
    for x, y in zip(*got):
        assert np.isfinite(x).all()
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)
