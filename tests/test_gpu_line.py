"""Runs of 1D systems in one launch (k_line) against the per-step kernels over
the forms the rule accepts, and against the oracle where it has them.

Bars: FP32 1e-5 and FP64 1e-12 rel-L2 against the per-step kernels (rounding of
two transform orders over a few steps), 1e-4 / 1e-10 against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O

from tests.parity import check_spectrum  # noqa: E402

pytestmark = pytest.mark.gpu
TWO = {"f32": 1e-5, "f64": 1e-12}
TOL = {"f32": 1e-4, "f64": 1e-10}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2405_02410_gb300 import build
    build.build()


def pss():
    from paper_2405_02410_gb300 import pss as m
    return m


def _run(n, prec, build, resident, batch=1, knobs=None):
    P = pss()
    s = P.System((n,), dt=0.01, seed=31, batch=batch, precision=prec, dx=(0.8,))
    nf = build(s)
    s.set_tuning("resident", resident)
    for b in range(batch):
        s.select_instance(b)
        for f in range(nf):
            s.init_uniform(f, -0.3, 0.3)
    l0 = s.launch_count
    s.step(7)
    launches = s.launch_count - l0
    s.step(4)
    out = []
    for b in range(batch):
        s.select_instance(b)
        out += [s.get_spectrum(f) for f in range(nf)]
    return out, launches


def _field(s, name, terms, noise=1, order=2, frame=None, lhs=((1.0, 0), (0.7, 1), (0.4, 2))):
    f = s.add_field(name)
    s.add_term(f, True, [(-1, c, p) for c, p in lhs], [(f, 1)])
    for mono, fac in terms:
        if len(fac) == 1:
            s.add_term(f, False, mono, [(f, fac[0])])
        else:
            s.add_product_term(f, mono, [(f,) + fac])
    if noise is not None:
        s.set_noise(f, s.add_param("D" + name, 0.05), noise)
    s.set_dealias(f, order)
    if frame:
        s.set_frame(f, *frame)
    return f


FORMS = {
    "cubic": lambda s: [_field(s, "a", [([(-1, -1.0, 1)], (3,))])] and 1,
    "quadratic_order0": lambda s: [_field(s, "a", [([(-1, -0.5, 0)], (2,))], noise=0, order=0)] and 1,
    "linear_noise2": lambda s: [_field(s, "a", [], noise=2)] and 1,
    "power1_quiet": lambda s: [_field(s, "a", [([(-1, 0.2, 0)], (1,))], noise=None, order=3)] and 1,
    "kpz": lambda s: [_field(s, "h", [([(-1, 0.5, 0)], (2, 0, 0))], noise=0)] and 1,
    "deriv_order0": lambda s: [_field(s, "h", [([(-1, 0.5, 1), (-1, 0.1, 0)], (1, 0, 1))], order=0)] and 1,
    "lap_power4": lambda s: [_field(s, "h", [([(-1, 0.1, 0)], (4, -1, 1))], order=3)] and 1,
    "degree4": lambda s: [_field(s, "a", [([(-1, -1.0, 1)], (3,))], lhs=((0.5, 1), (0.01, 4)))] and 1,
    "frame": lambda s: [_field(s, "a", [([(-1, -1.0, 0)], (3,))], noise=0, frame=(5, 0.5, -0.25))] and 1,
    "frame_linear": lambda s: [_field(s, "a", [], noise=None, frame=(32, 1.0, 0.0))] and 1,
    "two_fields": lambda s: [_field(s, "a", [([(-1, -1.0, 1)], (3,))]), _field(s, "b", [([(-1, 0.5, 0)], (2, 0, 0))], frame=(3, 0.1, 0.2))] and 2,
}


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n", [64, 256, 1024])
def test_agrees_with_the_per_step_kernels(n, form, prec):
    a, la = _run(n, prec, FORMS[form], 1, batch=3 if form == "two_fields" else 1)
    b, lb = _run(n, prec, FORMS[form], 0, batch=3 if form == "two_fields" else 1)
    assert la == 1 and lb >= 14
    for x, y in zip(a, b):
        assert np.linalg.norm(x - y) <= TWO[prec] * np.linalg.norm(y), np.linalg.norm(x - y) / np.linalg.norm(y)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", [64, 128, 512])
def test_matches_oracle(n, prec):
    kw = dict(dt=0.02, sigma=1.0, lam=0.6, D=0.02, seed=41)
    s = pss().kpz((n,), precision=prec, **kw)
    s.init_uniform(0, -0.5, 0.5)
    s.step(40)
    m = O.kpz((n,), **kw)
    check_spectrum(s.get_spectrum(0), O.half(O.run(m, O.to_spectrum(m, O.init_uniform(m, -0.5, 0.5)), 0, 40)), TOL[prec])
    kw = dict(dt=0.01, a=-1, b=1, K=1, D=0.05, seed=31)
    s = pss().model_b((n,), precision=prec, **kw)
    s.init_uniform(0, -0.2, 0.2)
    s.set_frame(0, 4, 0.3, -0.3)
    s.step(30)
    m = O.model_b((n,), **kw)
    ref = O.run_framed(m, O.to_spectrum(m, O.init_uniform(m, -0.2, 0.2)), 0, 30, 4, 0.3, -0.3)
    check_spectrum(s.get_spectrum(0), O.half(ref), TOL[prec])


def test_other_forms_keep_the_per_step_kernels():
    # a product of two fields, two product terms, a power beside a product, 32 sites
    P = pss()

    def launches(s):
        s.init_uniform(0, -0.1, 0.1)
        l0 = s.launch_count
        s.step(2)
        return s.launch_count - l0
    s = P.System((64,), dt=0.01, precision="f32")
    f, g = s.add_field("f"), s.add_field("g")
    s.add_product_term(f, [(-1, 0.1, 0)], [(f, 1), (g, 1)])
    assert launches(s) > 2
    s = P.kpz((64,), dt=0.01)
    s.add_term(0, False, [(-1, -0.3, 0)], [(0, 3)])
    assert launches(s) > 2
    assert launches(P.model_b((32,), dt=0.01)) > 2


def test_nonfinite_is_reported():
    P = pss()
    s = P.model_b((128,), noisy=False, precision="f32")
    x = np.zeros(128)
    x[4] = np.inf
    s.set_field(0, x)
    s.step(2)
    with pytest.raises(P.PssError) as ei:
        s.sync()
    assert ei.value.code == P.PSS_ENONFINITE


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", [64, 512, 1024])
def test_every_launch_of_a_linear_field_has_its_factors(n, prec):
    # no product, no noise: a step multiplies mode k by 1 / (1 + dt O(q_k)), and the
    # factors of a launch are read by other threads than the ones that made them; one
    # step per launch, so that each launch's first update counts.  Bar per step, in half
    # ulps: 16 of the denominator (q^2 carries 5, its square 10, coefficients 3, sums 3), 4
    # of the reciprocal, 1 of the product, 11 of the reference's own
    lhs = ((0.3, 0), (0.7, 1), (0.4, 2))
    s = pss().System((n,), dt=0.01, seed=3, precision=prec, dx=(0.8,))
    _field(s, "a", [], noise=None, lhs=lhs)
    x = np.random.default_rng(n).uniform(-1.0, 1.0, n).astype(s.rdtype)
    q2 = (2 * np.pi * np.arange(n // 2 + 1) / (n * 0.8)) ** 2
    g = 1.0 / (1.0 + 0.01 * sum(c * q2 ** p for c, p in lhs))
    tol = 64 * 32 * np.finfo(s.rdtype).eps / 2
    for _ in range(8):
        s.set_field(0, x)
        h0 = s.get_spectrum(0).astype(np.complex128)
        l0 = s.launch_count
        for _ in range(64):
            s.step(1)
        assert s.launch_count - l0 == 64
        h = s.get_spectrum(0)
        assert np.all(np.abs(h - h0 * g ** 64) <= tol * np.abs(h0 * g ** 64) + 1e-30)


@pytest.mark.parametrize("n", [64, 256, 1024])
def test_frame_adds_no_error_of_whole_transforms(n):
    # 100 steps of a heat bath in FP64 against extended precision with the step's own
    # factors 1 / (1 + dt q^2), rounded as the update takes them.  A step then rounds each
    # mode twice (the product, the frame's change), up to 2^-53 each: 100 steps that add up
    # as independent ones are sqrt(200 / 3) units, 9.1e-16; bar 1e-15, root mean square
    # over 16 initial fields
    ld = np.longdouble
    k = np.arange(n // 2 + 1) * (2 * np.pi / n)
    g = 1.0 / (1.0 + 0.5 * (k * k))
    err = 0.0
    for seed in range(16):
        x = np.random.default_rng(seed).uniform(4.5, 5.5, n)
        s = pss().System((n,), dt=0.5, seed=1, precision="f64")
        f = s.add_field("T")
        s.add_term(f, True, [(-1, 1.0, 1)], [(f, 1)])
        s.set_frame(f, 10, 10.0, 0.0)
        s.set_field(f, x)
        h = s.get_spectrum(f).astype(np.clongdouble)
        for _ in range(100):
            r = np.fft.irfft(h * g, n)
            r[:10], r[-10:] = 10, 0
            h = np.fft.rfft(r)
        s.step(100)
        got = np.fft.irfft(s.get_spectrum(f).astype(np.clongdouble), n)
        err += float(((got - r) ** 2).sum() / (r * r).sum()) / 16
    assert err <= 1e-15 ** 2, err ** 0.5


def test_an_explicit_term_added_after_a_captured_run():
    # a list with a system twice is captured, with the 1D run's explicit term among its
    # launch arguments: a term that is added later has to reach the next call
    P = pss()

    def make():
        s = P.System((64,), dt=0.01, seed=9, precision="f64")
        f = s.add_field("a")
        s.add_term(f, True, [(-1, 0.5, 1)], [(f, 1)])
        s.init_uniform(f, -0.5, 0.5)
        return s
    a, b = make(), make()
    P.step_many([a, a], 2)
    b.step(4)
    for s in (a, b):
        s.add_term(0, False, [(-1, -1.0, 0)], [(0, 3)])
    P.step_many([a, a], 2)
    b.step(4)
    np.testing.assert_array_equal(a.get_spectrum(0), b.get_spectrum(0))
