"""Forms a call's size selects: column blocks without a staging area (2048^2 float, 1024^2 double),
the persistent stepper's two forms, and feature buffers off a 16-byte boundary."""
import numpy as np
import pytest

import ttsh_inputs as ti
from oracle import ttsh_oracle as O

pytestmark = pytest.mark.gpu

# the parity tolerances of the other GPU tests: a few units in the last place through two
# transforms of each field a step
TOL = {64: 1e-12, 32: 1e-5}


@pytest.fixture(scope="module")
def T():
    from paper_2304_03306_gb300 import build, ttsh
    build.build()
    ttsh.load_library()
    return ttsh


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec,n", [(32, 2048), (64, 1024)])
def test_lean_column_pass_matches_oracle(T, prec, n):
    dx = 20.48 / n
    mask = ti.circle_mask(n, dx, 5.4)
    vx, vy = ti.noise_velocity(mask, 31, 0.3)
    p = O.Params(n=n, dx=dx)
    dft, idft = O.threaded_dft()
    K = O.process_mask(mask, dft=dft, idft=idft)
    s = O.project_velocity(vx, vy, p, dft=dft, idft=idft)
    for _ in range(2):
        s = O.step(s, K, p, dft=dft, idft=idft)
    d = T.Domain(mask, n, dx, precision=prec)
    d.set_velocity(vx, vy)
    d.step(2)
    gvx, gvy, _ = d.fields()
    w, _ = d.spectral_state()
    M = n // 4
    ref = np.concatenate([s.w_hat[: M + 1, : M + 1], s.w_hat[-M:, : M + 1]]).T
    assert rel(w, ref) <= TOL[prec]
    assert rel(np.stack([gvx, gvy]), np.stack([s.vx, s.vy])) <= TOL[prec]
    d.close()


@pytest.mark.parametrize("count", [4, 60])   # 65 items a step each: below and above the lean form's 3700
def test_persistent_forms_equal_single_domains_bit_for_bit(T, count):
    n, dx = 128, 0.16
    masks = [ti.circle_mask(n, dx, 5.0 + 0.02 * i) for i in range(count)]

    def make(i):
        d = T.Domain(masks[i], n, dx)
        d.init_noise(i, 0.3)
        return d

    doms = [make(i) for i in range(count)]
    b = T.Batch(doms)
    assert b.persistent
    b.step(37)
    b.synchronize()
    for i in (0, count // 2, count - 1):
        alone = make(i)
        alone.step(37)
        wa, va = alone.spectral_state()
        wb, vb = doms[i].spectral_state()
        assert np.array_equal(wa, wb) and np.array_equal(va, vb), i
        alone.close()
    b.close()
    for d in doms:
        d.close()


@pytest.mark.parametrize("prec", [32, 64])
def test_features_off_a_16_byte_boundary(T, prec):
    torch = pytest.importorskip("torch")
    n, dx = 64, 0.25
    d = T.Domain(ti.circle_mask(n, dx, 5.2), n, dx, precision=prec)
    d.init_noise(3, 0.3)
    net = T.FNO(n=n, width=32, modes=4, layers=1, max_batch=1, seed=0)
    scales = np.array([0.5, 2.0, 4.0, 0.25], np.float32)   # powers of two: exact
    net.set_scales(scales, 1.0)
    buf = torch.zeros(4 * n * n + 1, device="cuda")
    x = torch.zeros(4 * n * n, device="cuda")
    net.features(d, x.data_ptr())
    net.features(d, buf[1:].data_ptr())
    d.synchronize()
    assert torch.equal(x, buf[1:])
    vx, vy, w = d.fields()
    ref = np.stack([w, vx, vy, d.mask()], axis=-1).astype(np.float32) * scales
    assert np.array_equal(x.cpu().numpy().reshape(n, n, 4), ref)
    net.close()
    d.close()
