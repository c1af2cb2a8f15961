"""FP64 launches spread over the whole chip: single-column CTAs, radix 2 and 4,
and the table-driven normals, against the oracle at the edges of their
ranges."""
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


@pytest.mark.parametrize("shape", [(64,), (512, 4), (128, 64), (16, 8, 32)])
@pytest.mark.parametrize("power", [0, 1, 2, 3, 4])
def test_noise_increments(shape, power):
    # no operator, no product: one step from zero is the noise increment itself.
    # A normal is a few roundings of values up to 6 standard deviations: 16 units
    # of 2^-53 each bound it, 1.1e-14 of the mode's standard deviation
    P = pss()
    s = P.System(shape, dt=0.1, seed=77, precision="f64")
    f = s.add_field("phi")
    pD = s.add_param("D", 0.3)
    s.set_noise(f, pD, power)
    m = O.Model(shape=shape, dt=0.1, noise_D=0.3, noise_pow=power, noisy=True, seed=77)
    n = int(np.prod(shape))
    q = [2 * np.pi * np.fft.fftfreq(k) for k in shape[:-1]] + [2 * np.pi * np.arange(shape[-1] // 2 + 1) / shape[-1]]
    q2 = sum(g * g for g in np.meshgrid(*q, indexing="ij"))
    sd = np.sqrt(n * 0.3 * 0.1 * q2 ** power)
    for step in range(3):
        s.set_step(step)
        s.set_spectrum(f, np.zeros(s.half_shape, dtype=np.complex128))
        s.step(1)
        err = np.abs(s.get_spectrum(f) - O.half(O.noise(m, step)))
        assert np.all(err <= 1.1e-14 * 1.5 * sd), float((err / np.maximum(sd, 1e-300)).max())


# sides at the edges of the rules: 16 (first single-column side), radix 2 and 4
# (few and many transforms), 1024, self-paired pencils, ragged last tiles
@pytest.mark.parametrize("shape,order,steps", [
    ((16, 16), 2, 20), ((16, 1024), 3, 8), ((1024, 16), 2, 8), ((512, 512), 2, 3), ((8, 64), 0, 20),
    ((16, 4, 8), 2, 10), ((64, 4, 16), 3, 10), ((16, 128, 4), 0, 6), ((128, 16, 64), 2, 4), ((4, 512, 16), 2, 4),
    ((8, 1024, 4), 2, 3), ((1024, 4, 4), 2, 3), ((1024,), 2, 20), ((8,), 2, 20)])
def test_shapes_match_oracle(shape, order, steps):
    P = pss()
    s = P.System(shape, dt=0.005, seed=8, precision="f64")
    P.add_model_a_field(s, a=-1, b=1, K=1, D=0.05, name="psi", dealias_order=order)
    P.add_model_b_field(s, a=-1, b=1, K=1, D=0.05, name="phi", dealias_order=order)
    ms = [O.model_a(shape, dt=0.005, a=-1, b=1, K=1, D=0.05, seed=8, field_id=0, dealias_order=order),
          O.model_b(shape, dt=0.005, a=-1, b=1, K=1, D=0.05, seed=8, field_id=1, dealias_order=order)]
    for f in (0, 1):
        s.init_uniform(f, -0.1, 0.1)
    s.step(steps)
    for f, m in enumerate(ms):
        ref = O.half(O.run(m, O.to_spectrum(m, O.init_uniform(m, -0.1, 0.1)), 0, steps))
        check_spectrum(s.get_spectrum(f), ref, 1e-10, order=order, what=f"field {f}")
        check = np.fft.irfftn(ref, s=shape, axes=tuple(range(len(shape))))
        assert np.linalg.norm(s.get_field(f) - check) <= 1e-10 * np.linalg.norm(check)


def test_nonfinite_is_reported():
    P = pss()
    for bad in (np.inf, np.nan):
        s = P.model_b((32, 64), noisy=False, precision="f64")
        x = np.zeros((32, 64))
        x[3, 4] = bad
        s.set_field(0, x)
        s.step(2)
        with pytest.raises(P.PssError) as ei:
            s.sync()
        assert ei.value.code == P.PSS_ENONFINITE


@pytest.mark.parametrize("D,dt", [(1.0, 1.0), (0.05, 0.01)])
def test_normals_have_no_common_error(D, dt):
    # the relative error that all draws of a run share adds up over its steps, unlike
    # their independent roundings.  Projection of the increments' error on the increments,
    # in units of 2^-53: the 16 000 components' roundings (about 1 each) leave 0.01, the
    # 128 intervals' table entries (0.3 each, halved by the root) 0.02; bar 0.15
    ld = np.longdouble
    ny = nx = 128
    seed = 20240502
    s = pss().System((ny, nx), dt=dt, seed=seed, precision="f64")
    f = s.add_field("phi")
    s.set_noise(f, s.add_param("D", D), 0)
    s.step(1)
    got = s.get_spectrum(f)[:, 1:nx // 2]
    kx, ky = np.meshgrid(np.arange(1, nx // 2), np.arange(ny))
    hxe = nx // 2 + 2
    ctr = np.zeros((kx.size, 4), dtype=np.uint32)
    ctr[:, 0] = ((ky * hxe + kx) >> 1).reshape(-1)
    w = O.philox(ctr, np.tile(np.array([seed & 0xFFFFFFFF, seed >> 32], dtype=np.uint32), (kx.size, 1)))
    odd = (kx.reshape(-1) & 1) == 1
    u0, u1 = ((np.where(odd, w[:, 2 + i], w[:, i]) >> 8).astype(ld) + ld(0.5) for i in (0, 1))
    u0, u1 = u0 / 2 ** 24, u1 / 2 ** 24
    pi = 4 * np.arctan(ld(1))
    r = np.sqrt(-2 * np.log(u0)) * ld(np.sqrt(ny * nx * D * dt))
    re, im = r * np.cos(2 * pi * u1), r * np.sin(2 * pi * u1)
    er, ei = got.real.reshape(-1).astype(ld) - re, got.imag.reshape(-1).astype(ld) - im
    common = float((er * re + ei * im).sum() / (re * re + im * im).sum() * ld(2) ** 53)
    assert abs(common) <= 0.15, common


@pytest.mark.parametrize("shape", [(64,), (128, 128), (16, 512), (32, 16, 64)])
def test_whole_fields_take_radix_8_transforms(shape):
    # a field's way in and out is the radix-8 (y and z in 3D: 16) transform's, bit for bit,
    # whatever radix the steps' products take; the transforms of fewer roundings
    P = pss()
    x = np.random.default_rng(5).uniform(-1.0, 1.0, shape)
    out = []
    for radix in ({}, dict(row_radix=8, col_radix=16 if len(shape) == 3 else 8, mid_radix=16)):
        s = P.System(shape, dt=0.01, precision="f64")
        s.add_field("phi")
        for k, v in radix.items():
            s.set_tuning(k, v)
        s.set_field(0, x)
        h = s.get_spectrum(0)
        if out:
            s.set_spectrum(0, out[0][0])
        out.append((h, s.get_field(0)))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
