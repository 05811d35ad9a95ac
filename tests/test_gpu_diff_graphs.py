"""Repeated gradient calls: the second call of a shape in a row builds CUDA
graphs of its launches and later ones replay them.  Every call's results equal
those of a first call on a fresh context bit for bit, whatever was called
before."""
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


@pytest.mark.parametrize("T, K_ctg, limit", [(24, 3, None), (7, 9, None), (24, 2, 0), (130, 1, None), (1, 10, None)])
def test_repeated_calls_equal_first_calls(T, K_ctg, limit):
    from paper_2410_17203_gb300 import UnrolledCost
    case = make_case(scale_case(40, T, K_ctg, seed=90 + T, n_hvdc=1))
    rng = np.random.default_rng(5)

    def context():
        d = UnrolledCost(case, checkpoint_every=4)
        if limit is not None:
            d.set_record_limit(limit)
        return d

    kept = context()
    # (iterations, gradients): runs of one shape, a shape in between, and back
    for K, grads in [(9, True)] * 4 + [(9, False)] * 3 + [(6, True), (9, True), (9, True), (9, True)]:
        x = case["load_p"] * rng.lognormal(0.0, 0.1, size=case["load_p"].shape)
        u = case["line_u"] * rng.uniform(0.5, 1.0, size=case["line_u"].shape)
        fresh = context()
        f0, g0 = fresh.cost_grad(K, load_p=x, line_u=u, grads=grads)
        f1, g1 = kept.cost_grad(K, load_p=x, line_u=u, grads=grads)
        fresh.close()
        assert f0 == f1
        if grads:
            for k in g0:
                np.testing.assert_array_equal(g0[k], g1[k], err_msg=k)
    kept.close()
