"""The forms of the device phase against the oracle and against each other:
the register-resident inner ADMM at the edges of its chunks of steps per lane
and the shared-memory form beyond them, one device kernel or separate
averages and sums, one instance or a batch."""
import numpy as np
import pytest

from gridgen import make_case, scale_case
from helpers import compare_states
from oracle import Oracle, OracleOptions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2410_17203_gb300 import load_library
    load_library()


@pytest.mark.parametrize("T", [2, 31, 32, 63, 64, 127, 128, 159, 160, 255, 256])
def test_inner_chunks_match_oracle(T):
    """A battery holds T + 1 elements and a ramp-limited generator T: their
    chunk sizes change at T = 31 / 32, 63 / 64 and so on; 255 is the longest
    horizon in registers.  12 iterations include one change of the penalty."""
    from paper_2410_17203_gb300 import Solver
    case = make_case(scale_case(20, T, 2, seed=500 + T, stor_per_node=0.2, n_hvdc=1))
    opts = dict(adapt_every=10, eps=0.0)
    s = Solver(case, opts)
    s.iterate(12)
    o = Oracle(case, OracleOptions(**opts))
    o.iterate(12, stop=False)
    compare_states(s.state(), o)
    s.close()


@pytest.mark.parametrize("n, T, K, alpha", [
    (60, 1, 9, 1.0), (60, 31, 10, 1.0), (40, 128, 3, 1.0), (30, 255, 2, 1.5), (60, 7, 22, 1.5),
    # a line pass long enough to hide the devices: averages and device sums are kernels of their own
    (2600, 160, 24, 1.0), (2600, 160, 24, 1.5), (3000, 121, 24, 1.0),
])
def test_single_instance_and_batch_agree_bit_for_bit(n, T, K, alpha):
    """A batch forms every average where it is used, sums device powers in the
    node pass and takes horizons beyond 127 steps through shared memory."""
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(n, T, K, seed=7))
    opts = dict(adapt_every=10, eps=0.0, alpha=alpha)
    single, member = Solver(case, opts), Solver(case, opts)
    single.iterate(13)
    b = opf_batch_create([member.h])
    try:
        opf_batch_iterate(b, 13)
        x, y = single.state(), member.state()
        for k in x:
            np.testing.assert_array_equal(x[k], y[k], err_msg=k)
    finally:
        opf_batch_destroy(b)
        single.close()
        member.close()


@pytest.mark.parametrize("T", [24, 7])
def test_relaxed_split_launches_equal_one_launch(T):
    """The over-relaxed node pass without residual sums (all but the last
    iteration of a call and the adaptation iterations) gives the iterate of
    the pass with them bit for bit, wherever the calls end."""
    from paper_2410_17203_gb300 import Solver
    case = make_case(scale_case(90, T, 3, seed=41))
    opts = dict(adapt_every=10, eps=0.0, alpha=1.5)
    a, b = Solver(case, opts), Solver(case, opts)
    a.iterate(33)
    for n in (1, 1, 4, 9, 3, 15):
        b.iterate(n)
    x, y = a.state(), b.state()
    for k in x:
        np.testing.assert_array_equal(x[k], y[k], err_msg=k)
    a.close()
    b.close()


@pytest.mark.parametrize("T", [1, 2, 7, 24])
def test_inner_state_round_trip(T):
    """The inner-ADMM duals through opf_get_state / opf_set_state, host and
    device buffers: bit for bit the same, zero for a battery's equality rows'
    beta, and in the layout from which the oracle continues alike."""
    import torch
    from paper_2410_17203_gb300 import Solver, opf_get_state, opf_set_state, state_shapes
    case = make_case(scale_case(40, T, 2, seed=60 + T, stor_per_node=0.1))
    opts = dict(adapt_every=0, eps=0.0, rho_p=2.0)
    a, b, c = (Solver(case, opts) for _ in range(3))
    a.iterate(15)
    x = a.state()
    b.set_state(x)
    np.testing.assert_array_equal(b.state()["inner"], x["inner"])
    dev = {k: torch.from_numpy(v).cuda() for k, v in x.items()}
    opf_set_state(c.h, dev, on_device=True)
    out = {k: torch.full(s, np.nan, dtype=torch.float32, device="cuda") for k, s in state_shapes(c.info).items()}
    opf_get_state(c.h, on_device=True, out=out)
    np.testing.assert_array_equal(out["inner"].cpu().numpy(), x["inner"])
    nr, ns = a.info["n_ramp"] * 2 * (4 * T - 2), 8 * T + 4
    stor = x["inner"][nr:].reshape(a.info["n_stor"], 2, ns)
    assert not stor[:, 1, :2 * T + 2].any() and stor[:, 0].any()
    o = Oracle(case, OracleOptions(**opts))
    o.load_state(x)
    o.iterate(3, stop=False)
    for s in (b, c):
        s.iterate(3)
        compare_states(s.state(), o)
        s.close()
    a.close()


@pytest.mark.parametrize("n, T, K, alpha", [(30, 1, 5, 1.0), (20, 24, 2, 1.0), (12, 7, 1, 1.5), (2, 1, 0, 1.0), (20, 8, 2, 1.5)])
def test_small_instance_on_one_cta(n, T, K, alpha):
    """An instance without inner-ADMM devices that fits one CTA's rounds runs
    whole calls in one launch: iterates, residuals, penalties and the residual
    history equal those of the batch kernels bit for bit, over calls that end
    on and between residual iterations."""
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(n, T, K, seed=n + T, stor_per_node=0.0, ramp=False, fixed_frac=0.3,
                                n_hvdc=0, lines_per_node=1.3 if n > 2 else 0.5))
    opts = dict(adapt_every=10, eps=1e-9, check_every=7, alpha=alpha)
    a, b = Solver(case, opts), Solver(case, opts)
    assert a.info["kernels_per_iteration"] == 1
    h = opf_batch_create([b.h])
    try:
        for m in (1, 6, 13, 20, 1, 1060):
            a.iterate(m)
            opf_batch_iterate(h, m)
            x, y = a.state(), b.state()
            for k in x:
                np.testing.assert_array_equal(x[k], y[k], err_msg=k)
            np.testing.assert_array_equal(a.residuals(), b.residuals())
        np.testing.assert_array_equal(a.history(), b.history())
        i, j = a.get_info(), b.get_info()
        assert (i["iterations"], i["rho_p"], i["rho_theta"]) == (j["iterations"], j["rho_p"], j["rho_theta"])
        o = Oracle(case, OracleOptions(adapt_every=10, eps=0.0, alpha=alpha))
        o.iterate(30, stop=False)
        c = Solver(case, dict(adapt_every=10, eps=0.0, alpha=alpha))
        c.iterate(30)
        compare_states(c.state(), o)
        c.close()
    finally:
        opf_batch_destroy(h)
        a.close()
        b.close()
