"""Bounded device-side waits: what is left behind when one runs out.

Every wait in the kernels (the scanning router's exchange between its blocks, the waits of the summary
router's warps for one another, the grid barriers and the bulk-copy arrival of the fused anticipator build)
gives up after a number of polls.  The test hook pre_test_set_spin_limit makes that number small, with 0 the
first unsuccessful poll gives up: nothing faults or hangs, the kernels leave through their ordinary give-up path.  These tests check the
status and the state the header promises after that, against the oracle.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2504_03702_b200 import binding as B  # noqa: E402
from paper_2504_03702_b200 import workloads as W  # noqa: E402
from paper_2504_03702_b200.state import DeviceState  # noqa: E402
from tests.gpu_util import assert_scores_close, assert_state_equal, dev  # noqa: E402


@pytest.mark.parametrize("idx", [1, 2])
def test_router_wait_that_runs_out_keeps_a_routed_prefix(idx):
    wl = W.make_config(idx)
    st = DeviceState.from_workload(wl)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    n0 = wl.n_requests
    ap, ad = wl.ticks[0]
    ap, ad = ap[:256], ad[:256]

    st.select_router(B.ROUTE_SCAN)      # the kernel whose blocks wait for one another
    assert B.pre_test_set_spin_limit(st.ctx, 0) == B.PRE_OK
    choice, score = st.route_batch(dev(ap), dev(ad))
    assert st.status() == B.PRE_ETIMEOUT
    routed = st.sync_count() - n0
    assert 0 <= routed < len(ap), "with no patience at all the batch cannot have been finished"
    got_c, got_s = choice.cpu().numpy(), score.cpu().numpy()
    want_c, want_s = ref.route_batch(ap[:routed], ad[:routed])
    assert (got_c[:routed] == want_c).all()
    assert_scores_close(got_s[:routed], want_s, got_c[:routed])
    assert (got_c[routed:] == -1).all() and (got_s[routed:] == 0.0).all()
    assert_state_equal(st, ref, "after the wait ran out")

    # the context is still good: the rest of the batch, with the usual patience
    assert B.pre_test_set_spin_limit(st.ctx, 1 << 22) == B.PRE_OK
    choice, score = st.route_batch(dev(ap[routed:]), dev(ad[routed:]))
    assert st.status() == B.PRE_OK
    want_c, want_s = ref.route_batch(ap[routed:], ad[routed:])
    assert (choice.cpu().numpy() == want_c).all()
    assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert_state_equal(st, ref, "after the rest of the batch")
    st.close()


def test_admission_router_wait_that_runs_out():
    wl = W.make_config(1)
    st = DeviceState.from_workload(wl)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    n0 = wl.n_requests
    ap, ad = wl.ticks[0]
    ap, ad = ap[:128], ad[:128]
    st.make_queue(16)
    st.select_router(B.ROUTE_SCAN)      # the kernel whose blocks wait for one another
    B.pre_test_set_spin_limit(st.ctx, 0)
    _, choice, score = st.route_admit(dev(ap), dev(ad), overload_level=0.95, overload_share=0.10)
    assert st.status() == B.PRE_ETIMEOUT
    routed = st.sync_count() - n0
    got_c = choice.cpu().numpy()
    want_c, _ = ref.route_batch(ap[:routed], ad[:routed])      # nothing blocks at these levels
    assert (got_c[:routed] == want_c).all() and (got_c[routed:] == -1).all()
    assert st.queue_state.cpu().tolist() == [0, 0]
    assert_state_equal(st, ref, "after the wait ran out")
    st.close()


# (instances, steps, beta): all rows held by the deciding warp, in one launch and in three; lists; binary64 scores
SUMMARY_SHAPES = [(3, 64, 1.0), (8, 64, 1.0), (200, 96, 1.0), (600, 64, 1.0), (2100, 40, 1.0), (40, 700, 0.75), (600, 64, 0.75)]


def summary_case(n_inst, h, beta, seed):
    n, n_arr = 6 * n_inst, 400
    wl = W.make_random(seed, n_inst, h, n, 0, max_prompt=300, max_output=h, beta=beta)
    rng = np.random.default_rng(seed)
    ap = rng.integers(0, 300, n_arr).astype(np.int32)
    ad = np.where(rng.random(n_arr) < 0.2, rng.integers(1, 8, n_arr), rng.integers(8, 2 * h, n_arr)).astype(np.int32)
    ad[50::97] = 0                                      # malformed
    wl.max_requests = n + 2 * n_arr
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    return st, ref, n, ap, ad


@pytest.mark.parametrize("n_inst,h,beta", SUMMARY_SHAPES)
@pytest.mark.parametrize("polls", [0, 2, 20, 200])
def test_summary_router_wait_that_runs_out_keeps_a_routed_prefix(n_inst, h, beta, polls):
    st, ref, n0, ap, ad = summary_case(n_inst, h, beta, 31)
    # the rows that would be read if a decision that never reached the table were counted
    st.instance[n0:].fill_(2 ** 30)
    B.pre_test_set_spin_limit(st.ctx, polls)
    choice, score = st.route_batch(dev(ap), dev(ad))
    status = st.status()
    routed = st.sync_count() - n0
    ok = ad >= 1
    if polls == 0:
        assert status == B.PRE_ETIMEOUT and routed < ok.sum(), "with no patience at all the batch cannot have been finished"
    assert status in (B.PRE_ETIMEOUT, B.PRE_EBADREQ)
    end = int(np.flatnonzero(ok)[routed]) if routed < ok.sum() else len(ap)        # the first arrival that was not decided
    assert status == B.PRE_ETIMEOUT or end == len(ap)
    got_c, got_s = choice.cpu().numpy(), score.cpu().numpy()
    want_c, want_s = ref.route_batch(ap[:end], ad[:end])
    assert (got_c[:end] == want_c).all()
    assert_scores_close(got_s[:end], want_s, want_c)
    assert (got_c[end:] == -1).all() and (got_s[end:] == 0.0).all()
    assert_state_equal(st, ref, "after the wait ran out")

    # the context is still good: the rest of the batch, with the usual patience
    B.pre_test_set_spin_limit(st.ctx, 1 << 22)
    choice, score = st.route_batch(dev(ap[end:]), dev(ad[end:]))
    assert st.status() in (B.PRE_OK, B.PRE_EBADREQ)
    want_c, want_s = ref.route_batch(ap[end:], ad[end:])
    assert (choice.cpu().numpy() == want_c).all()
    assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert_state_equal(st, ref, "after the rest of the batch")
    st.close()


def test_warps_that_have_nothing_to_do_are_not_lost():
    """Arrivals of one token for which no list is asked for, and a long run of malformed ones that reach nobody: both take many
    times the limit, and nothing is owed to the warps that wait meanwhile."""
    n_inst, h = 900, 64
    n = 8 * n_inst
    wl = W.make_random(33, n_inst, h, n, 0, max_prompt=300, max_output=h)
    rng = np.random.default_rng(33)
    short, bad = 3000, 300000
    ap = rng.integers(0, 300, short + bad + 50).astype(np.int32)
    ad = np.ones(short + bad + 50, np.int32)
    ad[short:short + bad] = 0
    wl.max_requests = n + short + 50
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    B.pre_test_set_spin_limit(st.ctx, 4096)
    choice, score = st.route_batch(dev(ap), dev(ad))
    assert st.status() == B.PRE_EBADREQ, "a warp that waited for work gave the batch up"
    want_c, want_s = ref.route_batch(ap, ad, fast=True)
    assert (choice.cpu().numpy() == want_c).all()
    assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert_state_equal(st, ref)
    st.close()


@pytest.mark.parametrize("n_inst,h,beta", SUMMARY_SHAPES)
@pytest.mark.parametrize("polls", [0, 20])
def test_summary_admission_router_wait_that_runs_out(n_inst, h, beta, polls):
    """Waiting requests that were not reached keep their place, arrivals that were not reached are dropped."""
    st, ref, n0, ap, ad = summary_case(n_inst, h, beta, 32)
    ad = np.maximum(ad, 1)
    st.make_queue(128)
    head, waiting = 100, 70
    at = (head + np.arange(waiting)) % 128
    qp, qd = np.zeros(128, np.int32), np.zeros(128, np.int32)
    qp[at], qd[at] = ap[:waiting], ad[:waiting]
    st.queue_prompt.copy_(dev(qp)); st.queue_predicted.copy_(dev(qd))
    st.queue_state.copy_(torch.tensor([head, waiting]))
    st.instance[n0:].fill_(2 ** 30)
    B.pre_test_set_spin_limit(st.ctx, polls)
    qc, choice, score = st.route_admit(dev(ap[waiting:]), dev(ad[waiting:]), overload_level=50.0)     # nothing blocks at this level
    status = st.status()
    routed = st.sync_count() - n0
    assert status == B.PRE_ETIMEOUT and routed < len(ap) if polls == 0 else status in (B.PRE_ETIMEOUT, B.PRE_OK)
    assert status == B.PRE_ETIMEOUT or routed == len(ap)
    want_c, want_s = ref.route_batch(ap[:routed], ad[:routed])
    got = np.concatenate([qc[:waiting].cpu().numpy(), choice.cpu().numpy()])
    assert (got[:routed] == want_c).all()
    assert (got[routed:waiting] == -2).all() and (got[max(routed, waiting):] == -1).all()
    got_s = score.cpu().numpy()
    if routed > waiting:
        assert_scores_close(got_s[:routed - waiting], want_s[waiting:], want_c[waiting:])
    assert (got_s[max(routed - waiting, 0):] == 0.0).all()
    left = max(waiting - routed, 0)
    assert st.queue_state.cpu().tolist() == [(head + waiting - left) % 128, left]
    assert_state_equal(st, ref, "after the wait ran out")
    st.close()


def test_build_wait_that_runs_out_and_the_next_build():
    wl = W.make_config(2)
    st = DeviceState.from_workload(wl)
    ref = oracle.State.from_workload(wl)
    ref.anticipate()
    st.anticipate()                                   # a first build, so that the second one takes the quick layout
    assert st.status() == B.PRE_OK
    B.pre_test_set_spin_limit(st.ctx, 0)
    st.anticipate()                                   # the maps this leaves are undefined
    assert st.status() == B.PRE_ETIMEOUT
    B.pre_test_set_spin_limit(st.ctx, 1 << 22)
    for _ in range(2):                                # exact layout, then the learned one again
        st.curves.fill_(-1)
        st.anticipate()
        assert st.status() == B.PRE_OK
        assert (st.curves.cpu().numpy() == ref.curves).all()
        assert (st.current_d.cpu().numpy() == ref.current_d).all()
    st.close()
