"""Gradient contexts of several horizons side by side: creating or calling one
changes nothing for the others."""
import numpy as np
import pytest

from gridgen import make_case, scale_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2410_17203_gb300 import load_library
    load_library()


@pytest.mark.parametrize("T_long, T_short", [(168, 24), (140, 130), (168, 128)])
def test_a_shorter_context_leaves_a_longer_one_alone(T_long, T_short):
    """The shared-memory inner ADMM (beyond 127 steps) needs more than the
    default limit, which belongs to the kernel and not to a context."""
    from paper_2410_17203_gb300 import UnrolledCost
    long = UnrolledCost(make_case(scale_case(12, T_long, 1, seed=3, stor_per_node=0.2)), checkpoint_every=4)
    f0, g0 = long.cost_grad(4)
    short = UnrolledCost(make_case(scale_case(12, T_short, 1, seed=4, stor_per_node=0.2)), checkpoint_every=4)
    s0, _ = short.cost_grad(4)
    for _ in range(4):   # launched directly, as graphs are built, and replayed
        f, g = long.cost_grad(4)
        assert f == f0
        for k in g0:
            np.testing.assert_array_equal(g[k], g0[k], err_msg=k)
    assert short.cost_grad(4)[0] == s0
    long.close()
    short.close()


@pytest.mark.parametrize("T, K", [(1, 9), (3, 17), (4, 8), (7, 20), (8, 7), (8, 40), (9, 20)])
def test_short_horizons_with_many_contingencies(T, K):
    """Up to eight steps, eight lanes share a step's sum over contingencies:
    cost and gradients against the FP64 autograd reference, at the bounds of
    the other comparisons with it (about 1e-6 per step of FP32 rounding)."""
    from oracle.unrolled import Unrolled
    from paper_2410_17203_gb300 import UnrolledCost
    case = make_case(scale_case(150, T, K, seed=40 + T, stor_per_node=0.1, n_hvdc=1))
    ref = Unrolled(case, rho_p=10.0, rho_theta=20.0)
    prm = ref.params()
    f, _ = ref.run(prm, 12)
    f.backward()
    d = UnrolledCost(case, rho_p=10.0, rho_theta=20.0, checkpoint_every=5)
    for _ in range(4):   # launched directly, as graphs are built, and replayed
        cost, g = d.cost_grad(12)
        assert cost == pytest.approx(float(f.detach()), rel=1e-4)
        for k, v in prm.items():
            want = v.grad.numpy()
            assert np.linalg.norm(g[k] - want) <= 2e-3 * np.linalg.norm(want), k
    assert d.cost_grad(12, grads=False)[0] == cost
    d.close()
