"""A context iterated alone and as a member of a batch by turns: the same
iterates as one that only runs alone, whichever form of the inner ADMM each
call takes (registers up to 255 steps alone and up to 127 in a batch, shared
memory beyond)."""
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


def _assert_same_state(a, b):
    x, y = a.state(), b.state()
    for k in x:
        np.testing.assert_array_equal(x[k], y[k], err_msg=k)


@pytest.mark.parametrize("adapt_every", [0, 5])
@pytest.mark.parametrize("T", [127, 128, 168, 255, 256])
def test_alone_then_batch_by_turns(T, adapt_every):
    """The factors that one form leaves behind serve the other: fixed
    penalties (factored once, by the first call) and adapting ones."""
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(24, T, 2, seed=900 + T, stor_per_node=0.2))
    opts = dict(adapt_every=adapt_every, eps=0.0)
    ref, ctx = Solver(case, opts), Solver(case, opts)
    b = opf_batch_create([ctx.h])
    try:
        for alone, n in ((True, 3), (False, 4), (True, 5), (False, 6), (False, 1), (True, 2)):
            ref.iterate(n)
            if alone:
                ctx.iterate(n)
            else:
                opf_batch_iterate(b, n)
            _assert_same_state(ctx, ref)
    finally:
        opf_batch_destroy(b)
        ref.close()
        ctx.close()


@pytest.mark.parametrize("n, T, K, n_hvdc", [
    (40, 300, 4, 0), (40, 300, 4, 2), (30, 2048, 1, 1),   # one device kernel, no shared memory
    (2000, 100, 12, 2), (3000, 33, 22, 0),                # averages and device sums apart, beside the line pass
])
def test_instances_without_inner_admm_devices(n, T, K, n_hvdc):
    """Closed-form devices and links alone: every plan gives the batch's bits
    (one device kernel whatever the size), short ones also the oracle's."""
    from helpers import compare_states
    from oracle import Oracle, OracleOptions
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(n, T, K, seed=31 + T, stor_per_node=0.0, ramp=False, n_hvdc=n_hvdc))
    opts = dict(adapt_every=5, eps=0.0)
    single, member = Solver(case, opts), Solver(case, opts)
    single.iterate(12)
    b = opf_batch_create([member.h])
    try:
        opf_batch_iterate(b, 12)
        _assert_same_state(member, single)
        if n <= 40:
            o = Oracle(case, OracleOptions(**opts))
            o.iterate(12, stop=False)
            compare_states(single.state(), o)
    finally:
        opf_batch_destroy(b)
        single.close()
        member.close()


@pytest.mark.parametrize("T", [1000, 1015, 1023, 1024])
def test_batch_at_the_edge_of_48_kb(T):
    """A batch's device kernel takes 48 (T + 1) bytes of shared memory beside
    its own: the sum, not the former alone, decides whether it must ask for
    more than the default 48 KB.  The bits are those of the context alone."""
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(5, T, 0, seed=T, stor_per_node=0.2))
    opts = dict(adapt_every=0, eps=0.0)
    single, member = Solver(case, opts), Solver(case, opts)
    single.iterate(2)
    b = opf_batch_create([member.h])
    try:
        opf_batch_iterate(b, 2)
        _assert_same_state(member, single)
    finally:
        opf_batch_destroy(b)
        single.close()
        member.close()
