"""The cluster-resident FP32 2D step (tuning key "resident"): a run of steps as
one launch with every slot's state on chip, against the oracle, against the
per-step kernels over everything the rule that selects it accepts, and
against itself for every cluster size.

Bars: rel-L2 <= 1e-4 per mode against the FP64 oracle; rel-L2 <= 1e-5 against
the per-step kernels (FP32 rounding of two transform orders over a few steps);
bit for bit across cluster sizes and ways to take the steps.
"""
import numpy as np
import pytest

from oracle import oracle as O

from tests.parity import check_spectrum  # noqa: E402

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


def _system(shape, batch=1, fields=1, order=2, noisy=True, knobs=None, power=3, noise_pow=None):
    P = pss()
    s = P.System(shape, dt=0.01, seed=5, batch=batch, precision="f32", dx=(1.0, 0.7, 1.0))
    for i in range(fields):
        f = s.add_field(f"f{i}")
        pa, pD = s.add_param(f"a{i}", -0.8), s.add_param(f"D{i}", 0.05)
        # fields take turns: conserved with a fourth-order operator, non-conserved
        up = 1 if i % 2 == 0 else 0
        s.add_term(f, True, [(pa, 1.0, up), (-1, 1.0, 1 + up)] + ([(-1, 0.01, 3)] if i == 1 else []), [(f, 1)])
        if power:
            s.add_term(f, False, [(-1, -1.0, up)], [(f, power)])
        if noisy:
            s.set_noise(f, pD, up if noise_pow is None else noise_pow)
        s.set_dealias(f, order)
    for k, v in (knobs or {}).items():
        s.set_tuning(k, v)
    for b in range(batch):
        s.select_instance(b)
        for f in range(fields):
            s.init_uniform(f, -0.2, 0.2)
    return s


def _spectra(s, fields):
    out = []
    for b in range(s.batch):
        s.select_instance(b)
        out += [s.get_spectrum(f) for f in range(fields)]
    return np.stack(out)


def _launches(s, n):
    l0 = s.launch_count
    s.step(n)
    return s.launch_count - l0


SHAPES = [(32, 32), (64, 64), (128, 128), (32, 512), (512, 32), (64, 256), (256, 128), (512, 128), (128, 64)]


@pytest.mark.parametrize("batch,fields,order,kw", [
    (1, 1, 2, {}), (3, 2, 3, {}), (2, 1, 0, {}), (1, 2, 2, dict(noisy=False)), (1, 1, 2, dict(power=2)),
    (1, 1, 2, dict(power=0)), (1, 1, 2, dict(power=1, noise_pow=2)), (1, 1, 2, dict(noise_pow=3))])
@pytest.mark.parametrize("shape", SHAPES)
def test_agrees_with_the_per_step_kernels(shape, batch, fields, order, kw):
    a = _system(shape, batch, fields, order, **kw)
    b = _system(shape, batch, fields, order, knobs=dict(resident=0), **kw)
    assert _launches(a, 7) == 1 and _launches(b, 7) >= 14
    a.step(5)
    b.step(5)
    x, y = _spectra(a, fields), _spectra(b, fields)
    for u, v in zip(x, y):
        assert np.linalg.norm(u - v) <= 1e-5 * np.linalg.norm(v)
    assert a.get_step() == b.get_step() == 12


@pytest.mark.parametrize("shape,batch", [((64, 64), 1), ((128, 128), 3), ((512, 128), 1), ((32, 256), 2), ((256, 256), 32)])
def test_cluster_sizes_and_run_lengths_give_the_same_bits(shape, batch):
    ref = _system(shape, batch)
    ref.step(9)
    want = _spectra(ref, 1)
    for c in (1, 2, 4, 8, 16):
        s = _system(shape, batch, knobs=dict(res_ctas=c))
        s.step(4)
        s.step(5)
        assert _spectra(s, 1).tobytes() == want.tobytes(), c
    if shape != (256, 256):
        m = _system(shape, batch)
        other = _system((64, 128), 2)
        slow = _system((512, 256), 1)       # per-step kernels, from a graph beside the resident runs
        pss().step_many([other, m, slow], 9)
        assert _spectra(m, 1).tobytes() == want.tobytes()
        alone = _system((512, 256), 1)
        alone.step(9)
        assert _spectra(slow, 1).tobytes() == _spectra(alone, 1).tobytes()


@pytest.mark.parametrize("shape,order", [((32, 64), 2), ((256, 32), 3), ((128, 128), 2), ((128, 512), 2)])
def test_matches_oracle(shape, order):
    kw = dict(dt=0.01, a=-1, b=1, K=1, D=0.05, seed=17, dealias_order=order)
    s = pss().model_b(shape, precision="f32", **kw)
    s.init_uniform(0, -0.1, 0.1)
    assert _launches(s, 40) == 1
    m = O.model_b(shape, **kw)
    ref = O.half(O.run(m, O.to_spectrum(m, O.init_uniform(m, -0.1, 0.1)), 0, 40))
    check_spectrum(s.get_spectrum(0), ref, 1e-4)


def test_256_batch_agrees_with_the_two_kernel_step():
    a, b = _system((256, 256), 32), _system((256, 256), 32, knobs=dict(resident=0))
    assert _launches(a, 6) == 1 and _launches(b, 6) >= 12
    x, y = _spectra(a, 1), _spectra(b, 1)
    for u, v in zip(x, y):
        assert np.linalg.norm(u - v) <= 1e-5 * np.linalg.norm(v)


def test_switching_paths_and_changing_parameters_mid_run():
    shape = (64, 128)
    a, b = _system(shape, 2), _system(shape, 2, knobs=dict(resident=0))
    for s in (a, b):
        s.step(5)
        s.set_param_batch(0, np.array([-0.5, -1.1]))
        s.step(5)
    a.set_tuning("resident", 0)
    a.step(5)
    a.set_tuning("resident", 1)
    a.step(5)
    b.step(10)
    x, y = _spectra(a, 1), _spectra(b, 1)
    assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)


def test_nonfinite_state_is_reported():
    P = pss()
    s = _system((64, 32), noisy=False)
    x = np.zeros((64, 32), dtype=np.float32)
    x[3, 5] = np.inf
    s.set_field(0, x)
    s.step(2)
    with pytest.raises(P.PssError) as ei:
        s.sync()
    assert ei.value.code == P.PSS_ENONFINITE


@pytest.mark.parametrize("first", [0, 1])
def test_step_many_leaves_every_system_as_it_was_when_a_capture_fails(first):
    # a system of the list whose launch the host refuses (its radix-8 columns of 1024 points
    # take too many threads), found while its graph is captured: nothing of the list runs
    P = pss()
    res = P.model_b((64, 64), dt=0.01, a=-1, b=1, K=1, D=0.05, seed=4, precision="f32")
    bad = P.model_b((1024, 4, 4), dt=0.001, a=-1, b=1, K=1, D=0.05, seed=4, precision="f64")
    systems = [res, bad] if first == 0 else [bad, res]
    for s in systems:
        s.init_uniform(0, -0.1, 0.1)
    P.step_many(systems, 2)
    before = [s.get_spectrum(0) for s in systems]
    bad.set_tuning("col_radix", 8)
    for _ in range(2):
        with pytest.raises(P.PssError):
            P.step_many(systems, 20)
        for s, x in zip(systems, before):
            assert s.get_step() == 2
            np.testing.assert_array_equal(s.get_spectrum(0), x)
    bad.set_tuning("col_radix", 0)
    P.step_many(systems, 20)
    for s in systems:
        assert s.get_step() == 22
    twin = P.model_b((64, 64), dt=0.01, a=-1, b=1, K=1, D=0.05, seed=4, precision="f32")
    twin.init_uniform(0, -0.1, 0.1)
    twin.step(22)
    np.testing.assert_array_equal(res.get_spectrum(0), twin.get_spectrum(0))
