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


@pytest.mark.parametrize("alpha", [1.0, 1.5])
def test_members_equal_contexts_alone_in_every_bit(alpha):
    """Iterates, residuals, penalties and histories of a batch's instances are
    those of each context alone, whatever CTAs the node kernel deals them: with
    every instance running, after some have stopped (on tolerances of their
    own), after compaction, after a reset, and in every layout.  The largest
    has more node items than its grid has threads, the smallest less than one
    CTA's worth; eleven are more than half of what stops."""
    from paper_2410_17203_gb300 import (Solver, opf_batch_autotune, opf_batch_compact, opf_batch_create,
                                        opf_batch_destroy, opf_batch_iterate, opf_reset)
    sizes = [(3000, 24, 10), (5, 1, 0), (300, 24, 4), (60, 7, 22), (200, 1, 9), (90, 31, 2), (40, 12, 3),
             (700, 48, 1), (25, 128, 1), (50, 24, 20), (30, 300, 0)]
    cases = [make_case(scale_case(n, T, K, seed=70 + i, n_hvdc=i % 2 if n > 20 else 0))
             for i, (n, T, K) in enumerate(sizes)]
    # all but three stop at the first stopping test that finds residuals below a generous tolerance
    opts = [dict(adapt_every=5, check_every=4, alpha=alpha, history_len=64, eps=1e-9 if i in (0, 3, 7) else 1.0)
            for i in range(len(sizes))]
    alone = [Solver(c, o) for c, o in zip(cases, opts)]
    member = [Solver(c, o) for c, o in zip(cases, opts)]

    def check():
        for a, m in zip(alone, member):
            _assert_same_state(m, a)
            np.testing.assert_array_equal(m.residuals(), a.residuals())
            np.testing.assert_array_equal(m.history(), a.history())
            i, j = a.get_info(), m.get_info()
            assert [i[k] for k in ("iterations", "converged", "rho_p", "rho_theta")] == \
                   [j[k] for k in ("iterations", "converged", "rho_p", "rho_theta")]

    def both(n):
        for a in alone:
            if not a.get_info()["converged"]:
                a.iterate(n)
        opf_batch_iterate(b, n)
        check()

    b = opf_batch_create([m.h for m in member])
    try:
        for n in (3, 9, 20):
            both(n)
        left = sum(not a.get_info()["converged"] for a in alone)
        assert left == opf_batch_compact(b)
        both(7)
        for h in [a.h for a in alone] + [m.h for m in member]:
            opf_reset(h)
        opf_batch_autotune(b, steps=2)
        for n in (2, 17):
            both(n)
    finally:
        opf_batch_destroy(b)
        for s in alone + member:
            s.close()


@pytest.mark.parametrize("T", [256, 700, 1400])
def test_staged_horizons_match_oracle(T):
    """Batteries and ramp-limited generators staged in shared memory by four,
    two and one warps to a CTA, over a change of the penalty, alone and in a
    batch beside a short instance."""
    from helpers import compare_states
    from oracle import Oracle, OracleOptions
    from paper_2410_17203_gb300 import Solver, opf_batch_create, opf_batch_destroy, opf_batch_iterate
    case = make_case(scale_case(6, T, 1, seed=T, stor_per_node=0.2, lines_per_node=1.2))
    short = make_case(scale_case(30, 24, 2, seed=5))
    opts = dict(adapt_every=5, eps=0.0)
    single, member, beside, ref = Solver(case, opts), Solver(case, opts), Solver(short, opts), Solver(short, opts)
    single.iterate(7)
    ref.iterate(7)
    b = opf_batch_create([beside.h, member.h])
    try:
        opf_batch_iterate(b, 7)
        _assert_same_state(member, single)
        _assert_same_state(beside, ref)
        o = Oracle(case, OracleOptions(**opts))
        o.iterate(7, stop=False)
        assert o.rho_p != OracleOptions(**opts).rho_p
        compare_states(single.state(), o)
    finally:
        opf_batch_destroy(b)
        for s in (single, member, beside, ref):
            s.close()
