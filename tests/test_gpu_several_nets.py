"""Networks of different shapes alive at once: they share kernels, not each other's limits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2304_03306_gb300 import build, ttsh
    build.build()
    ttsh.load_library()
    return ttsh


# The first network of each row launches with more shared memory than a later one: the layer kernels
# (fewer modes, fewer points, a smaller ring of columns), and the separate kernels of an odd mode
# count and of more than 16 modes.
@pytest.mark.parametrize("first,later", [((256, 16), [(256, 4), (64, 4)]), ((256, 16), [(512, 16)]),
                                         ((128, 16), [(16, 4)]), ((512, 3), [(32, 3)]), ((256, 32), [(128, 18)])])
def test_a_network_works_after_others_are_made(T, first, later):
    torch = pytest.importorskip("torch")
    n, m = first
    net = T.FNO(n=n, width=32, modes=m, layers=2, max_batch=1, seed=3)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((n, n, 4), device="cuda", generator=g)
    t = torch.randn((n, n), device="cuda", generator=g)
    torch.cuda.synchronize()

    def outputs():
        y = torch.zeros((n, n), device="cuda")
        torch.cuda.synchronize()
        net.forward(x.data_ptr(), y.data_ptr(), 1)
        loss, grad = net.loss_grad(x.data_ptr(), t.data_ptr(), 1, want_grad=True)
        torch.cuda.synchronize()
        return y.cpu().numpy(), loss, grad

    before = outputs()
    others = [T.FNO(n=k, width=32, modes=mm, layers=1, max_batch=1, seed=4) for k, mm in later]
    after = outputs()
    assert np.array_equal(before[0], after[0]) and before[1] == after[1] and np.array_equal(before[2], after[2])
    for o in others + [net]:
        o.close()
