"""ttsh_step_noalloc in several calls equals one call, bit for bit."""
import numpy as np
import pytest

import ttsh_inputs as ti

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2304_03306_gb300 import build, ttsh
    build.build()
    ttsh.load_library()
    return ttsh


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512])
def test_split_calls_equal_one_call(T, prec, n):
    torch = pytest.importorskip("torch")
    dx = 20.48 / n
    dom = T.Domain(ti.circle_mask(n, dx, 5.2), n, dx, precision=prec)
    dom.init_noise(n, 0.3)
    w, v = dom.spectral_state()
    dt = torch.float32 if prec == 32 else torch.float64
    K = torch.tensor(dom.mask(), dtype=dt, device="cuda").contiguous()
    dom.close()
    p = T.ttsh_default_params(n=n, dx=dx, precision=prec)

    def run(calls):
        w_d = torch.tensor(np.stack([w.real, w.imag], axis=-1), dtype=dt, device="cuda").contiguous()
        v_d = torch.tensor(v, dtype=dt, device="cuda").contiguous()
        torch.cuda.synchronize()
        for k in calls:
            T.ttsh_step_noalloc(p, K.data_ptr(), w_d.data_ptr(), v_d.data_ptr(), k)
        torch.cuda.synchronize()
        return w_d.cpu().numpy(), v_d.cpu().numpy()

    whole = run([12])
    for calls in ([6, 6], [1, 4, 7]):
        split = run(calls)
        assert np.array_equal(whole[0], split[0]) and np.array_equal(whole[1], split[1]), calls
