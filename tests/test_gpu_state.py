"""Checkpoint and resume through the C ABI (pss_save_state / pss_load_state).

A run saved in the middle and loaded into a fresh handle takes the same steps,
bit for bit, as the run that was never interrupted: on the FP32 2D path with
the noise drawn a step ahead, on the generic kernels (1D, 3D, FP64), on a
batched system with per-instance parameters, and across parameter changes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2405_02410_gb300 import build
    build.build()


def P():
    from paper_2405_02410_gb300 import pss
    return pss


def _spectra(s, nfields):
    out = []
    for b in range(s.batch):
        s.select_instance(b)
        out.extend(s.get_spectrum(f) for f in range(nfields))
    s.select_instance(0)
    return out


def _model_b(shape, prec="f32", batch=1, seed=2405):
    pss = P()
    s = pss.System(shape, dt=0.01, seed=seed, precision=prec, batch=batch)
    pss.add_model_b_field(s, a=-1, b=1, K=1, D=0.01)
    return s


@pytest.mark.parametrize("shape,prec,path", [
    ((256, 256), "f32", "persist2d"),
    ((512, 256), "f32", "fast2d"),
    ((64, 64), "f32", "generic"),
    ((8, 16, 32), "f64", "generic"),
    ((1024,), "f32", "generic"),
])
def test_resume_is_bit_identical(shape, prec, path):
    a = _model_b(shape, prec)
    assert a.step_path == path, a.step_path
    a.init_uniform(0, -0.1, 0.1)
    a.step(7)
    blob = a.save_state()
    a.step(13)
    ref = a.get_spectrum(0)
    b = _model_b(shape, prec, seed=99)        # a different seed: the state carries the saved one
    b.load_state(blob)
    assert b.get_step() == 7
    b.step(13)
    got = b.get_spectrum(0)
    assert got.tobytes() == ref.tobytes()
    a.close()
    b.close()


def test_resume_of_a_batch_with_per_instance_parameters():
    shape, batch = (256, 256), 3
    a = _model_b(shape, batch=batch)
    a.set_param_batch(0, np.array([-1.2, -0.9, -0.6]))        # "phi.a" per instance
    for i in range(batch):
        a.select_instance(i)
        a.init_uniform(0, -0.1, 0.1)
    a.select_instance(0)
    a.step(5)
    blob = a.save_state()
    a.step(11)
    ref = _spectra(a, 1)
    b = _model_b(shape, batch=batch, seed=7)                   # default parameters and other seeds
    b.load_state(blob)
    assert abs(b.get_param(0) - (-1.2)) == 0.0
    b.step(11)
    got = _spectra(b, 1)
    for x, y in zip(got, ref):
        assert x.tobytes() == y.tobytes()


def test_two_fields_3d_and_the_step_counter():
    pss = P()
    shape = (8, 16, 16)

    def build(seed):
        s = pss.System(shape, dt=0.005, seed=seed, precision="f32")
        pss.add_model_a_field(s, a=-1, b=1, K=1, D=0.05, name="psi")
        pss.add_model_b_field(s, a=-1, b=1, K=1, D=0.05, name="phi")
        return s

    a = build(5)
    a.init_uniform(0, -0.05, 0.05)
    a.init_uniform(1, -0.05, 0.05)
    a.step(4)
    blob = a.save_state()
    a.step(9)
    b = build(6)
    b.load_state(blob)
    b.step(9)
    assert b.get_step() == a.get_step() == 13
    for f in (0, 1):
        assert b.get_spectrum(f).tobytes() == a.get_spectrum(f).tobytes()


def test_load_rejects_another_system_and_leaves_it_unchanged():
    pss = P()
    a = _model_b((64, 64))
    a.init_uniform(0, -0.1, 0.1)
    blob = a.save_state()
    b = _model_b((64, 128))
    b.init_uniform(0, -0.2, 0.2)
    before = b.get_spectrum(0)
    with pytest.raises(pss.PssError) as ei:
        b.load_state(blob)
    assert ei.value.code == pss.PSS_EINVAL
    assert b.get_spectrum(0).tobytes() == before.tobytes()
    with pytest.raises(pss.PssError):
        a.load_state(blob[:-8])                                 # truncated
    with pytest.raises(pss.PssError):
        a.load_state(b"not a state" + blob[11:])                # wrong tag
    c = _model_b((64, 64), prec="f64")
    with pytest.raises(pss.PssError):
        c.load_state(blob)                                      # other precision


@pytest.mark.parametrize("shape,prec", [((64, 64), "f32"), ((8, 512), "f32"), ((16, 8, 32), "f32"), ((64,), "f32"),
                                        ((32, 64), "f64"), ((4,), "f32"), ((4, 8, 4), "f64")])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_device_buffers_at_any_address(shape, prec, offset):
    # fields and spectra go in and out where they are in device memory: from an address of any
    # alignment (an element, not a vector) the same bits as through host memory, and not a
    # value beside the buffer is touched
    import torch
    pss = P()
    n = int(np.prod(shape))
    rng = np.random.default_rng(n + offset)
    x = rng.uniform(-1.0, 1.0, shape)
    host, dev = (pss.model_b(shape, dt=0.01, seed=2, precision=prec) for _ in range(2))
    x = x.astype(host.rdtype)
    host.set_field(0, x)
    buf = torch.full((n + 8,), 7.0, dtype=torch.float64 if prec == "f64" else torch.float32, device="cuda")
    buf[offset:offset + n] = torch.from_numpy(x.reshape(-1)).cuda()
    torch.cuda.synchronize()
    dev.set_field(0, buf[offset:offset + n].view(shape))
    want = host.get_spectrum(0)
    np.testing.assert_array_equal(dev.get_spectrum(0), want)
    out = torch.full_like(buf, 5.0)
    torch.cuda.synchronize()
    dev.get_field(0, out=out[offset:offset + n].view(shape))
    o = out.cpu().numpy()
    np.testing.assert_array_equal(o[offset:offset + n].reshape(shape), host.get_field(0))
    assert (o[:offset] == 5.0).all() and (o[offset + n:] == 5.0).all()
    m = want.size
    hb = torch.full((m + 8,), 3.0, dtype=torch.complex128 if prec == "f64" else torch.complex64, device="cuda")
    torch.cuda.synchronize()
    dev.get_spectrum(0, out=hb[offset:offset + m].view(want.shape))
    h = hb.cpu().numpy()
    np.testing.assert_array_equal(h[offset:offset + m].reshape(want.shape), want)
    assert (h[:offset] == 3.0).all() and (h[offset + m:] == 3.0).all()
    other = pss.model_b(shape, dt=0.01, seed=2, precision=prec)
    other.set_spectrum(0, hb[offset:offset + m].view(want.shape))
    np.testing.assert_array_equal(other.get_spectrum(0), want)


@pytest.mark.parametrize("shape,prec", [((64, 64), "f32"), ((16, 8, 32), "f64"), ((64,), "f32")])
def test_buffers_that_are_not_the_devices_own_are_copied(shape, prec):
    # a pointer passed as device memory that is pinned memory of the host: no kernel works on
    # it, the copies find its place
    import ctypes
    import torch
    pss = P()
    x = np.random.default_rng(3).uniform(-1.0, 1.0, shape)
    host, dev = (pss.model_b(shape, dt=0.01, seed=2, precision=prec) for _ in range(2))
    x = x.astype(host.rdtype)
    host.set_field(0, x)
    pin = torch.from_numpy(x.copy()).pin_memory()
    out = torch.zeros_like(pin).pin_memory()
    h = torch.zeros(host.half_shape, dtype=torch.complex128 if prec == "f64" else torch.complex64).pin_memory()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert pss.lib.pss_set_field(dev._h, 0, ptr(pin), pss.PSS_DEVICE) == pss.PSS_OK
    np.testing.assert_array_equal(dev.get_spectrum(0), host.get_spectrum(0))
    assert pss.lib.pss_get_field(dev._h, 0, ptr(out), pss.PSS_DEVICE) == pss.PSS_OK
    np.testing.assert_array_equal(out.numpy(), host.get_field(0))
    assert pss.lib.pss_get_spectrum(dev._h, 0, ptr(h), pss.PSS_DEVICE) == pss.PSS_OK
    np.testing.assert_array_equal(h.numpy(), host.get_spectrum(0))
    other = pss.model_b(shape, dt=0.01, seed=2, precision=prec)
    assert pss.lib.pss_set_spectrum(other._h, 0, ptr(h), pss.PSS_DEVICE) == pss.PSS_OK
    np.testing.assert_array_equal(other.get_spectrum(0), host.get_spectrum(0))
