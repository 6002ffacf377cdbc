"""The routing kernel that works on per-row summaries, on the inputs that take its special paths.

Every case is compared with the oracle's literal router decision by decision; the cases are built
so that a particular path of the kernel is certain to run: rows whose summary only bounds the peak
(scanned cell by cell), the same row winning several arrivals in a row (a decision has to wait for
a fold), whole-number and binary64 scores, every fold-thread layout, and the hand-over to the
scanning kernel when a value could leave 32 bits or the instances do not fit shared memory.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_03702_b200 import workloads as W

pytestmark = pytest.mark.gpu

from gpu_util import assert_scores_close, assert_state_equal, dev  # noqa: E402
from paper_2504_03702_b200 import binding as B  # noqa: E402
from paper_2504_03702_b200.state import DeviceState  # noqa: E402


def route_and_compare(wl, ap, ad, path=B.ROUTE_SUMMARY, batches=1):
    st = DeviceState.from_workload(wl)
    if path is not None:
        st.select_router(path)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    cuts = np.linspace(0, len(ap), batches + 1).astype(int)
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        choice, score = st.route_batch(dev(ap[lo:hi]), dev(ad[lo:hi]))
        want_c, want_s = ref.route_batch(ap[lo:hi], ad[lo:hi])
        got = choice.cpu().numpy()
        assert (got == want_c).all(), f"first difference at arrival {lo + int(np.argmax(got != want_c))}"
        assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert_state_equal(st, ref)
    assert st.status() == B.PRE_OK
    st.close()
    return ref


def rising_maps(seed, n_inst, h, n, beta=1.0, capacity=None):
    """Requests with short prompts that all outlast the window: every map rises with the step, the
    largest cell + step sits at the last step, and no arrival's ramp reaches it."""
    wl = W.make_random(seed, n_inst, h, n, 0, max_prompt=4, max_output=8, capacity=capacity, beta=beta)
    wl.predicted[:] = 3 * h + 5
    wl.generated[:] = np.arange(n, dtype=np.int32) % 7
    return wl


@pytest.mark.parametrize("beta,t_mem", [(1.0, 0.8), (2.0, 0.8), (0.75, 0.8), (1.0, 0.81237)])
def test_rows_that_are_only_bounded_are_scanned(beta, t_mem):
    wl = rising_maps(51, 37, 96, 900, beta=beta, capacity=40000)
    wl.t_mem = t_mem
    rng = np.random.default_rng(5)
    ap = rng.integers(0, 3000, 300).astype(np.int32)
    ad = rng.integers(1, 96, 300).astype(np.int32)      # every ramp ends before the last step
    wl.max_requests = 900 + 300
    before = oracle.State.from_workload(wl)
    before.anticipate()
    top = before.curves + np.arange(96)[None, :]
    assert (top.argmax(axis=1) == 95).all(), "the maps were meant to peak at the end of the window"
    route_and_compare(wl, ap, ad)


@pytest.mark.parametrize("beta", [1.0, 0.5])
def test_bounded_and_exact_rows_mixed(beta):
    """Half of the instances hold rising maps, the other half ordinary ones; short and long arrivals."""
    a = rising_maps(52, 20, 64, 400, beta=beta, capacity=30000)
    b = W.make_random(53, 20, 64, 400, 0, max_prompt=200, max_output=150, capacity=30000, beta=beta)
    wl = a
    wl.prompt = np.concatenate([a.prompt, b.prompt])
    wl.generated = np.concatenate([a.generated, b.generated])
    wl.predicted = np.concatenate([a.predicted, b.predicted])
    wl.instance = np.concatenate([a.instance, b.instance + 20]).astype(np.int32)
    wl.n_instances = 40
    rng = np.random.default_rng(6)
    ap = rng.integers(0, 500, 400).astype(np.int32)
    ad = np.where(rng.random(400) < 0.5, rng.integers(1, 4, 400), rng.integers(1, 300, 400)).astype(np.int32)
    wl.max_requests = 800 + 400
    route_and_compare(wl, ap, ad, batches=3)


@pytest.mark.parametrize("n_inst", [1, 2, 3, 5])
@pytest.mark.parametrize("beta", [1.0, 0.3])
def test_the_same_rows_win_again_and_again(n_inst, beta):
    """Few instances: a row that has just received an arrival is often the best one for the next."""
    wl = W.make_random(60 + n_inst, n_inst, 48, 60, 0, max_prompt=50, max_output=90, beta=beta)
    rng = np.random.default_rng(7)
    ap = rng.integers(0, 40, 500).astype(np.int32)
    ad = rng.integers(1, 120, 500).astype(np.int32)
    wl.max_requests = 60 + 500
    route_and_compare(wl, ap, ad, batches=2)


def test_one_almost_empty_instance_takes_a_long_run_of_arrivals():
    wl = W.make_random(70, 12, 80, 3000, 0, max_prompt=400, max_output=200)
    keep = wl.instance != 4
    keep[:3] = True
    for name in ("prompt", "generated", "predicted", "instance"):
        setattr(wl, name, getattr(wl, name)[keep])
    rng = np.random.default_rng(8)
    ap = rng.integers(1, 30, 600).astype(np.int32)
    ad = rng.integers(1, 60, 600).astype(np.int32)
    wl.max_requests = len(wl.prompt) + 600
    ref = route_and_compare(wl, ap, ad)
    assert (ref.instance[len(wl.prompt):len(wl.prompt) + 50] == 4).mean() > 0.5


@pytest.mark.parametrize("h", [1, 2, 7, 255, 1024, 1025, 2048, 2050, 4096, 4099, 8192])
def test_every_fold_layout(h):
    """Horizons on both sides of each cells-per-thread step, even and odd."""
    wl = W.make_random(80 + h % 50, 9, h, 150, 0, max_prompt=300, max_output=2 * h + 5)
    rng = np.random.default_rng(9)
    ap = rng.integers(0, 300, 120).astype(np.int32)
    ad = rng.integers(1, 2 * h + 5, 120).astype(np.int32)
    wl.max_requests = 150 + 120
    route_and_compare(wl, ap, ad)


def test_malformed_arrivals_and_a_full_table_on_the_summary_kernel():
    wl = W.make_random(90, 30, 32, 400, 0)
    rng = np.random.default_rng(10)
    ap = rng.integers(0, 60, 200).astype(np.int32)
    ad = rng.integers(1, 50, 200).astype(np.int32)
    ad[[0, 33, 64, 65, 199]] = 0
    ap[[31, 32, 100]] = -1
    wl.max_requests = 400 + 170
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    choice, score = st.route_batch(dev(ap), dev(ad))
    want_c, want_s = ref.route_batch(ap, ad)
    assert (choice.cpu().numpy() == want_c).all()
    assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert (score.cpu().numpy()[want_c < 0] == 0.0).all()
    assert_state_equal(st, ref)
    assert st.status() == B.PRE_ECAPACITY
    choice, _ = st.route_batch(dev(ap[:5]), dev(ad[:5]))          # the table is full now
    assert (choice.cpu().numpy() == -1).all()
    st.close()


def test_values_that_could_leave_32_bits_go_to_the_scanning_kernel():
    """The summary kernel declines the batch on the device; the result is the scanning kernel's."""
    wl = W.make_random(91, 25, 40, 3000, 0, max_prompt=2 ** 22, max_output=60, capacity=10 ** 9)
    rng = np.random.default_rng(11)
    ap = rng.integers(2 ** 26, 2 ** 27, 80).astype(np.int32)       # 80 such prompts can add 2^33 to a cell
    ad = rng.integers(1, 80, 80).astype(np.int32)
    wl.max_requests = 3000 + 80
    route_and_compare(wl, ap, ad)
    wl = W.make_random(92, 25, 40, 3000, 0, max_prompt=2 ** 27, max_output=60, capacity=10 ** 11)   # cells above 2^32 already
    wl.max_requests = 3000 + 80
    route_and_compare(wl, (ap // 1000).astype(np.int32), ad)


def test_whole_number_scores_that_could_reach_2_to_the_30_go_to_the_scanning_kernel():
    """beta and theta are whole numbers, so the context gets the whole-number kind of the summary kernel; with
    beta = 4096 and peaks around 2^19 the score bound passes 2^30 and the kernel declines on the device."""
    wl = W.make_random(97, 25, 40, 600, 0, max_prompt=2 ** 16, max_output=60, capacity=10 ** 5, beta=4096.0)
    rng = np.random.default_rng(15)
    ap = rng.integers(2 ** 12, 2 ** 14, 120).astype(np.int32)
    ad = rng.integers(1, 80, 120).astype(np.int32)
    wl.max_requests = 600 + 120
    ref = route_and_compare(wl, ap, ad)
    assert ref.curves.max() * 4096.0 > 2.0 ** 30, "the case was meant to pass the whole-number bound"


@pytest.mark.parametrize("n_inst,h", [(5, 16), (40, 900), (300, 24)])
def test_scores_beyond_binary64(n_inst, h):
    """A penalty coefficient of 1e308: a row that pays has an infinite score, and when all rows do, the first one wins with it."""
    wl = W.make_random(98, n_inst, h, 4 * n_inst, 0, max_prompt=200, max_output=h, capacity=2000, beta=1e308)
    rng = np.random.default_rng(16)
    n_arr = 8 * n_inst
    ap = rng.integers(50, 400, n_arr).astype(np.int32)
    ad = rng.integers(1, 2 * h, n_arr).astype(np.int32)
    wl.max_requests = 4 * n_inst + n_arr
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    choice, score = st.route_batch(dev(ap), dev(ad))
    want_c, want_s = ref.route_batch(ap, ad)
    assert np.isfinite(want_s[0]) and np.isinf(want_s[-1]), "the case was meant to run from finite scores to infinite ones"
    assert (choice.cpu().numpy() == want_c).all()
    assert (score.cpu().numpy() == want_s).all()
    assert_state_equal(st, ref)
    assert st.status() == B.PRE_OK
    st.close()


def test_selecting_the_kernel():
    wl = W.make_random(93, 20000, 4, 100, 0)
    st = DeviceState.from_workload(wl)
    assert B.pre_route_select(st.ctx, B.ROUTE_SUMMARY) == B.PRE_ESIZE       # too many instances for one block
    assert B.pre_route_select(st.ctx, 3) == B.PRE_EINVAL
    assert B.pre_route_select(st.ctx, -1) == B.PRE_EINVAL
    assert B.pre_route_select(st.ctx, B.ROUTE_SCAN) == B.PRE_OK
    assert B.pre_route_select(st.ctx, B.ROUTE_AUTO) == B.PRE_OK
    assert B.pre_route_select(None, B.ROUTE_AUTO) == B.PRE_EINVAL
    st.close()
    wl = W.make_random(94, 300, 16, 2000, 0)
    rng = np.random.default_rng(12)
    ap = rng.integers(0, 100, 300).astype(np.int32)
    ad = rng.integers(1, 40, 300).astype(np.int32)
    wl.max_requests = 2300
    for path in (B.ROUTE_AUTO, B.ROUTE_SCAN, B.ROUTE_SUMMARY):
        route_and_compare(wl, ap, ad, path=path)


def test_many_instances_with_binary64_scores_take_the_scanning_kernel():
    """More than 5,120 instances give a score lane more rows than the binary64 kind of the summary kernel
    keeps in registers: selecting that kernel outright is refused, the default routes with the other."""
    wl = W.make_random(96, 6000, 8, 20000, 0, max_prompt=100, max_output=20, beta=0.75)
    st = DeviceState.from_workload(wl)
    assert B.pre_route_select(st.ctx, B.ROUTE_SUMMARY) == B.PRE_ESIZE
    st.close()
    rng = np.random.default_rng(14)
    ap = rng.integers(0, 100, 200).astype(np.int32)
    ad = rng.integers(1, 20, 200).astype(np.int32)
    wl.max_requests = 20200
    route_and_compare(wl, ap, ad, path=B.ROUTE_AUTO)
    wl.beta = 2.0      # whole-number scores: the summary kernel takes this many instances
    route_and_compare(wl, ap, ad, path=B.ROUTE_SUMMARY)


def test_many_instances_close_to_the_shared_memory_limit():
    wl = W.make_random(95, 9300, 8, 30000, 0, max_prompt=100, max_output=20)
    rng = np.random.default_rng(13)
    ap = rng.integers(0, 100, 400).astype(np.int32)
    ad = rng.integers(1, 20, 400).astype(np.int32)
    wl.max_requests = 30400
    route_and_compare(wl, ap, ad)


@pytest.mark.parametrize("n_inst", [40, 700, 2100])
@pytest.mark.parametrize("path", [B.ROUTE_SUMMARY, B.ROUTE_SCAN])
def test_equal_scores_go_to_the_lowest_index(n_inst, path):
    """Empty instances and identical arrivals: every score is shared by many rows, in the same lane, in
    other lanes of the warp and in other warps, and the lowest index among them has to win each time
    (Sec. 4.3.3 names no tie rule; the oracle's argmin takes the first)."""
    wl = W.make_random(3, n_inst, 64, 0, 0, capacity=100000)
    n = 3 * n_inst + 17
    ap = np.full(n, 10, dtype=np.int32)
    ad = np.full(n, 5, dtype=np.int32)
    wl.max_requests = n
    ref = route_and_compare(wl, ap, ad, path=path)
    assert ref.instance[:n].tolist() == [k % n_inst for k in range(n)]


def test_streaming_ticks_on_both_kernels():
    """Route, step, route ... over the first ticks of the streaming configuration, both kernels in turn."""
    wl = W.make_config(4, n_ticks=4)
    st = DeviceState.from_workload(wl)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    for t, (ap, ad) in enumerate(wl.ticks):
        st.select_router(B.ROUTE_SUMMARY if t % 2 == 0 else B.ROUTE_SCAN)
        st.step()
        ref.step()
        choice, score = st.route_batch(dev(ap), dev(ad))
        want_c, want_s = ref.route_batch(ap, ad, fast=True)
        assert (choice.cpu().numpy() == want_c).all(), f"tick {t}"
        assert_scores_close(score.cpu().numpy(), want_s, want_c)
    assert_state_equal(st, ref)
    st.close()


@pytest.mark.parametrize("beta,level", [(1.0, 0.7), (0.75, 0.7), (0.4, 0.5)])
def test_admission_queue_on_the_summary_kernel(beta, level):
    """Several calls with a queue that fills and drains, whole-number and binary64 scores, the kernel selected outright."""
    wl = W.make_random(96, 5, 24, 120, 0, max_prompt=200, max_output=60, beta=beta)
    wl.max_requests = 120 + 400
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    st.make_queue(12)
    ref.make_queue(12)
    rng = np.random.default_rng(14)
    seen = set()
    for call in range(10):
        a = int(rng.integers(0, 40))
        ap = rng.integers(0, 200, a).astype(np.int32)
        ad = rng.integers(1, 60, a).astype(np.int32)
        if a > 3 and call % 3 == 1:
            ad[1] = 0                                   # malformed
        waiting = int(ref.queue_state[1])
        qc, c, s = st.route_admit(dev(ap), dev(ad), overload_level=level, overload_share=0.10)
        wqc, wc, ws = ref.route_admit(ap, ad, overload_level=level, overload_share=0.10)
        assert (c.cpu().numpy() == wc).all(), f"call {call}: arrivals"
        assert (qc[:waiting].cpu().numpy() == wqc).all(), f"call {call}: waiting requests"
        assert_scores_close(s.cpu().numpy(), ws, wc)
        assert st.queue_state.cpu().tolist() == ref.queue_state.tolist()
        assert_state_equal(st, ref, f"after call {call}")
        seen.update(np.unique(wc).tolist())
        seen.update((-10 - v for v in np.unique(wqc).tolist() if v >= 0))
        st.status()
        for _ in range(int(rng.integers(0, 4))):
            st.step()
            ref.step()
    assert -2 in seen and -3 in seen and any(v >= 0 for v in seen) and any(v <= -10 for v in seen), \
        "the case was meant to route, queue, turn away and route out of the queue"
    st.close()


@pytest.mark.parametrize("n_inst,h,n_arr", [(1, 32768 // 4, 9), (64, 512, 128), (64, 512, 129), (65, 504, 70), (128, 40, 300),
                                            (129, 65, 300), (256, 64, 400), (257, 63, 400), (2048, 9, 300), (2049, 70, 300),
                                            (257, 63, 24), (2049, 70, 12), (2500, 128, 25)])
@pytest.mark.parametrize("beta", [1.0, 0.75])
def test_both_sides_of_every_layout_of_the_deciding_warp(n_inst, h, n_arr, beta):
    """One launch or three, ramps by the routing block or by the whole grid, one to eight rows per lane, all rows or a list."""
    wl = W.make_random(500 + n_inst % 97, n_inst, h, 12 * n_inst, 0, max_prompt=300, max_output=2 * h + 9, beta=beta)
    rng = np.random.default_rng(20)
    ap = rng.integers(0, 300, n_arr).astype(np.int32)
    ad = rng.integers(1, 2 * h + 9, n_arr).astype(np.int32)
    wl.max_requests = 12 * n_inst + n_arr
    route_and_compare(wl, ap, ad, batches=2)


@pytest.mark.parametrize("n_inst,h", [(3, 700), (40, 900), (300, 260)])
@pytest.mark.parametrize("beta", [1.0, 0.5])
@pytest.mark.parametrize("queue", [False, True])
def test_rows_whose_largest_cell_moves_beyond_the_first_steps(n_inst, h, beta, queue):
    """Long requests with short prompts on maps that fall slowly: the bounds of the later steps overtake the first ones again
    and again, rows are brought up to date in the middle of a batch, turn full and near again, and are counted cell by cell."""
    n = 4 * n_inst
    wl = W.make_random(520 + n_inst % 7, n_inst, h, n, 0, max_prompt=6000, max_output=h, beta=beta)
    wl.generated[:] = 0
    rng = np.random.default_rng(21)
    n_arr = 900
    ap = np.where(rng.random(n_arr) < 0.3, rng.integers(2000, 6000, n_arr), rng.integers(0, 40, n_arr)).astype(np.int32)
    ad = np.where(rng.random(n_arr) < 0.4, rng.integers(1, 70, n_arr), rng.integers(h // 2, 2 * h, n_arr)).astype(np.int32)
    wl.max_requests = n + n_arr
    st = DeviceState.from_workload(wl)
    st.select_router(B.ROUTE_SUMMARY)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    if queue:
        st.make_queue(50)
        ref.make_queue(50)
    for lo in range(0, n_arr, 300):
        p, d = ap[lo:lo + 300], ad[lo:lo + 300]
        if queue:
            _, c, s = st.route_admit(dev(p), dev(d), overload_level=2.0, overload_share=0.3)
            _, wc, ws = ref.route_admit(p, d, overload_level=2.0, overload_share=0.3)
        else:
            c, s = st.route_batch(dev(p), dev(d))
            wc, ws = ref.route_batch(p, d)
        got = c.cpu().numpy()
        assert (got == wc).all(), f"first difference at arrival {lo + int(np.argmax(got != wc))}"
        assert_scores_close(s.cpu().numpy(), ws, wc)
        assert_state_equal(st, ref, f"after arrival {lo + 300}")
        st.step()
        ref.step()
    assert st.status() == B.PRE_OK
    st.close()


@pytest.mark.parametrize("n_inst,h,beta", [(2, 500, 1.0), (3, 901, 0.75), (280, 400, 1.0)])
def test_rows_brought_up_to_date_late_in_a_long_batch(n_inst, h, beta):
    """Runs of requests that leave a row's largest cell among the first steps, more of them than a warp has lanes, between requests
    that move it far out: the row then gets all ramps that its map lacks at once, several times in one batch."""
    n = 6 * n_inst
    wl = W.make_random(540 + n_inst, n_inst, h, n, 0, max_prompt=50, max_output=30, beta=beta, capacity=20000)
    rng = np.random.default_rng(22)
    ap, ad = [], []
    for run in (45 * n_inst, 20 * n_inst, 70 * n_inst) if n_inst < 10 else (5 * n_inst, 4 * n_inst):
        ap += [rng.integers(300, 900, run), rng.integers(0, 3, 12 * n_inst if n_inst < 10 else 3 * n_inst)]
        ad += [rng.integers(40, 64, run), rng.integers(h - 40, 2 * h, len(ap[-1]))]
    ap, ad = np.concatenate(ap).astype(np.int32), np.concatenate(ad).astype(np.int32)
    wl.max_requests = n + len(ap)
    route_and_compare(wl, ap, ad)


def case_of(kind):
    """Services on which summaries say little: empty ones, few requests per instance, all of them young, one-token arrivals."""
    n_inst, h, per, beta = {"empty": (512, 512, 0, 1.0), "empty, binary64": (2000, 300, 0, 0.75), "few": (600, 700, 4, 1.0),
                            "few, binary64": (600, 700, 4, 0.75), "young": (600, 700, 16, 1.0), "one token": (1024, 512, 64, 1.0)}[kind]
    wl = W.make_random(560 + n_inst % 89, n_inst, h, per * n_inst, 0, max_prompt=2000, max_output=h + h // 2, beta=beta,
                       capacity=None if per else 500001)
    if kind == "young":
        wl.generated[:] = 0
    rng = np.random.default_rng(23)
    ap = rng.integers(1, 2000, 1500).astype(np.int32)
    ad = rng.integers(1, h + h // 2, 1500).astype(np.int32)
    if kind == "one token":
        ad[:] = 1
    wl.max_requests = per * n_inst + 1500
    return wl, ap, ad


@pytest.mark.parametrize("kind", ["empty", "empty, binary64", "few", "few, binary64", "young", "one token"])
def test_the_default_is_not_slower_than_the_scanning_kernel(kind):
    """The library's choice against the kernel that reads every cell for every arrival, whose time does not depend on the rows: the best
    of five calls each, with half as much again as room (the two differ by less than 2 % from call to call)."""
    wl, ap, ad = case_of(kind)
    st = DeviceState.from_workload(wl)
    p, d = dev(ap), dev(ad)
    best, choices = {}, {}
    for path in (B.ROUTE_AUTO, B.ROUTE_SCAN):
        st.select_router(path)
        times = []
        for _ in range(5):
            st.n_requests.fill_(len(wl.prompt))
            st.queued_p.zero_()
            st.anticipate(len(wl.prompt))
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            choice, _ = st.route_batch(p, d)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        best[path], choices[path] = min(times), choice.cpu().numpy()
    assert (choices[B.ROUTE_AUTO] == choices[B.ROUTE_SCAN]).all()
    assert best[B.ROUTE_AUTO] <= 1.5 * best[B.ROUTE_SCAN], best
    st.close()


@pytest.mark.parametrize("beta", [1.0, 0.75])
@pytest.mark.parametrize("queue", [False, True])
def test_small_shapes_whose_numbers_leave_32_bits_against_expectation(beta, queue):
    """A small capacity promises small numbers, and one launch without the scanning kernel behind it; the maps hold cells above 2^32 all the
    same, and the routing block takes the batch cell by cell."""
    wl = W.make_random(99, 25, 40, 3000, 0, max_prompt=2 ** 27, max_output=60, capacity=1000, beta=beta)
    rng = np.random.default_rng(17)
    ap = rng.integers(2 ** 16, 2 ** 24, 80).astype(np.int32)
    ad = rng.integers(1, 80, 80).astype(np.int32)
    wl.max_requests = 3000 + 80
    if not queue:
        route_and_compare(wl, ap, ad)
        return
    st = DeviceState.from_workload(wl)
    ref = oracle.State.from_workload(wl)
    st.anticipate()
    ref.anticipate()
    st.make_queue(30)
    ref.make_queue(30)
    level = float(np.sort(ref.curves.max(axis=1))[-3]) / 1000
    for lo in (0, 40):
        qc, c, s = st.route_admit(dev(ap[lo:lo + 40]), dev(ad[lo:lo + 40]), overload_level=level, overload_share=0.0)
        wqc, wc, ws = ref.route_admit(ap[lo:lo + 40], ad[lo:lo + 40], overload_level=level, overload_share=0.0)
        assert (c.cpu().numpy() == wc).all() and (qc[:len(wqc)].cpu().numpy() == wqc).all()
        assert_scores_close(s.cpu().numpy(), ws, wc)
        assert st.queue_state.cpu().tolist() == ref.queue_state.tolist()
    assert_state_equal(st, ref)
    st.close()


@pytest.mark.parametrize("beta", [1000.5, 1e5 + 0.5, 1e9 + 0.25, 1e15])
@pytest.mark.parametrize("n_inst,h", [(40, 900), (300, 80), (2100, 30)])
def test_large_fractional_penalties(n_inst, h, beta):
    """Keys in units of several tokens: rows within the rounding are compared in binary64."""
    wl = W.make_random(580 + n_inst % 89, n_inst, h, 10 * n_inst, 0, max_prompt=3000, max_output=h, beta=beta)
    rng = np.random.default_rng(24)
    ap = rng.integers(1, 3000, 500).astype(np.int32)
    ad = rng.integers(1, 2 * h, 500).astype(np.int32)
    wl.max_requests = 10 * n_inst + 500
    route_and_compare(wl, ap, ad, batches=2)


@pytest.mark.parametrize("n_inst,h", [(7, 48), (40, 300), (140, 64), (257, 90), (2100, 40)])
@pytest.mark.parametrize("beta,capacity,t_mem", [(1.0, 1281, 0.8), (1.0, 5003, 0.8), (1.0, 40001, 0.8), (1.0, 20000, 0.812345),
                                                 (0.75, 2003, 0.8), (0.75, 30002, 0.8), (0.5, 9001, 0.8), (3.0, 7007, 0.8)])
def test_scores_with_a_fraction_that_all_paying_rows_share(n_inst, h, beta, capacity, t_mem):
    """beta a small dyadic fraction and a fractional threshold: whole-number keys decide as the binary64 scores do, ties among rows that pay and ties among
    rows that do not; peaks so far beyond the threshold (the small capacities) that beta times the excess is no longer exact."""
    wl = W.make_random(640 + n_inst % 83, n_inst, h, 10 * n_inst, 0, max_prompt=600, max_output=h, capacity=capacity, beta=beta)
    wl.t_mem = t_mem
    rng = np.random.default_rng(25)
    ap = rng.choice([40, 41, 300, 2000], 500).astype(np.int32)      # (many equal sums)
    ad = rng.choice([3, 30, h - 1, 2 * h], 500).astype(np.int32)
    wl.max_requests = 10 * n_inst + 500
    route_and_compare(wl, ap, ad, batches=2)


def one_request_each(prompt, generated, predicted, horizon, capacity, beta, arrivals):
    """One request per instance: the map of instance i rises from prompt + generated to its last step, where cell + step is largest."""
    n_inst = len(prompt)
    wl = W.make_random(1, n_inst, horizon, 0, 0, capacity=capacity, beta=beta)
    wl.prompt, wl.generated, wl.predicted = (np.asarray(x, dtype=np.int32) for x in (prompt, generated, predicted))
    wl.instance = np.arange(n_inst, dtype=np.int32)
    wl.max_requests = n_inst + arrivals
    return wl


def test_a_short_arrival_on_a_row_whose_top_costs_more_than_half_the_range_of_the_keys():
    """beta = 100,000: the top of row 150 lies at step 20, and its cells there cost 4 million less than cell + step says."""
    prompt, predicted = np.full(200, 999), np.full(200, 2)
    prompt[150], predicted[150] = 974, 22
    wl = one_request_each(prompt, np.ones(200), predicted, 128, 1000, 1e5, 1)
    ref = route_and_compare(wl, np.array([1], np.int32), np.array([2], np.int32))
    assert ref.instance[200] == 150, "the case was meant to go to the row with the far lower peak"


@pytest.mark.parametrize("n_inst", [20, 50, 100, 200])
@pytest.mark.parametrize("h", [40, 128])
@pytest.mark.parametrize("beta", [17000.0, 1e5, 1e6, 200.5, 2000.5, 1e15])
def test_short_arrivals_with_large_penalties(n_inst, h, beta):
    """Peaks within 20 tokens of the threshold, tops at steps up to 60 and as far above it: what such an arrival adds to the key of the
    top is less than any key holds.  Every sixth row has its top among the first steps, where most arrivals reach it."""
    rng = np.random.default_rng(int(beta) % 1000 + n_inst + h)
    step = rng.integers(5, min(h, 61), n_inst)
    step[::6] = rng.integers(0, 3, len(step[::6]))
    peak = 200 + rng.integers(-20, 21, n_inst)
    wl = one_request_each(peak - step - 1, np.ones(n_inst), step + 2, h, 250, beta, 60)
    ap, ad = rng.integers(0, 5, 60).astype(np.int32), rng.integers(1, 5, 60).astype(np.int32)
    before = oracle.State.from_workload(wl)
    before.anticipate()
    assert ((before.curves + np.arange(h)[None, :]).argmax(axis=1) == step).all() and (before.curves.max(axis=1) == peak).all()
    route_and_compare(wl, ap, ad, batches=3)


def skewed(n_inst, h, per, n_arr, beta, whole=True):
    """`per` requests per instance on average, assigned by Zipf: most instances hold a few requests, and the tops of many maps lie far out."""
    n = n_inst * per
    prompt, generated, predicted = W._lengths(77, n, 1024, 1.2, 16, 8192, 384, 1.2, 1, 4096, in_flight=True)
    instance = W._zipf_instances(77, n, n_inst, 1.1)
    wl = W.make_random(77, n_inst, h, 0, 0, beta=beta, capacity=W._capacity(prompt, generated, instance, n_inst) // 5 * 5 + (0 if whole else 3))
    wl.prompt, wl.generated, wl.predicted, wl.instance = prompt, generated, predicted, instance
    ap, _, ad = W._lengths(78, n_arr, 1024, 1.2, 16, 8192, 384, 1.2, 1, 4096, in_flight=False)
    wl.max_requests = n + n_arr
    return wl, ap, ad


@pytest.mark.parametrize("n_inst,h", [(300, 228), (700, 500), (1054, 228), (2100, 100)])
@pytest.mark.parametrize("beta,whole", [(1.0, True), (1.0, False), (0.75, False), (0.4, False)])
def test_far_rows_of_a_list_are_compared_in_place(n_inst, h, beta, whole):
    wl, ap, ad = skewed(n_inst, h, 20, 400, beta, whole)
    before = oracle.State.from_workload(wl)
    before.anticipate()
    far = (before.curves + np.arange(h)[None, :]).argmax(axis=1) >= 32
    assert far.mean() > 0.1 and not far.all(), "the case was meant to have far rows and others"
    route_and_compare(wl, ap, ad, batches=2)


def share_of_the_scanning_time(wl, ap, ad):
    """The library's choice of kernel against the scanning kernel, whose time does not depend on the rows: best of seven calls each."""
    st = DeviceState.from_workload(wl)
    p, d = dev(ap), dev(ad)
    best = {}
    for path in (B.ROUTE_AUTO, B.ROUTE_SCAN):
        st.select_router(path)
        times = []
        for _ in range(7):
            st.n_requests.fill_(len(wl.prompt))
            st.queued_p.zero_()
            st.anticipate(len(wl.prompt))
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            st.route_batch(p, d)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        best[path] = min(times)
    assert st.status() == B.PRE_OK
    st.close()
    return best[B.ROUTE_AUTO] / best[B.ROUTE_SCAN]


@pytest.mark.parametrize("beta,whole", [(1.0, True), (1.0, False)])
def test_arrivals_on_far_rows_do_not_take_a_look_at_all_rows(beta, whole):
    """Some 0.4 of the scanning kernel's time where a far row that wins is compared among the list's rows, 0.7 and more where each such
    arrival takes a look at all rows."""
    assert share_of_the_scanning_time(*skewed(1054, 228, 35, 817, beta, whole)) < 0.6


@pytest.mark.parametrize("n_inst", [4, 5, 20, 32, 33])
@pytest.mark.parametrize("beta,whole", [(1.0, True), (0.75, False)])
def test_small_services_with_a_long_backlog(n_inst, beta, whole):
    """Both sides of the rule that leaves the folds to the deciding warp, and of that for exact keys."""
    wl, ap, ad = skewed(n_inst, 57, 32, 900, beta, whole)
    route_and_compare(wl, ap, ad, batches=2)


@pytest.mark.parametrize("beta,whole", [(1.0, True), (0.75, False)])
def test_backlogs_of_small_services_are_folded_by_the_folding_warps(beta, whole):
    """32 rows, 2,000 arrivals: 0.05 to 0.07 of the scanning kernel's time, 0.13 to 0.17 with every fold made by the deciding warp itself; the limit lies
    half as much again above the one and below the other."""
    assert share_of_the_scanning_time(*skewed(32, 256, 128, 2000, beta, whole)) < 0.1


def long_prompts(n_inst, n_arr, beta, whole, median, sigma, longest):
    """Log-normal prompts up to `longest` on 512 steps, 64 requests per instance."""
    n = 64 * n_inst
    prompt, generated, predicted = W._lengths(79, n, median, sigma, 16, longest, 384, 1.2, 1, 4096, in_flight=True)
    instance = W._uniform_instances(79, n, n_inst)
    wl = W.make_random(79, n_inst, 512, 0, 0, beta=beta, capacity=W._capacity(prompt, generated, instance, n_inst) // 5 * 5 + (0 if whole else 3))
    wl.prompt, wl.generated, wl.predicted, wl.instance = prompt, generated, predicted, instance
    ap, _, ad = W._lengths(80, n_arr, median, sigma, 16, longest, 384, 1.2, 1, 4096, in_flight=False)
    wl.max_requests = n + n_arr
    return wl, ap, ad


LONG = {"half of the prompts beyond exact keys": (0.75, False, 65536, 1.2, 131072), "peaks far beyond the threshold": (0.75, False, 300, 2.0, 131072),
        "large penalty": (100.0, True, 1024, 1.2, 8192), "larger penalty": (700.0, True, 60, 1.2, 1500)}


@pytest.mark.parametrize("kind", LONG)
@pytest.mark.parametrize("n_inst", [3, 40, 100, 200, 300, 1100])
def test_batches_that_do_not_fit_exact_keys(kind, n_inst):
    """Whole-number scores and those of fractional thresholds, routed with rounded keys or a shorter list; and where few arrivals are too long, with exact ones."""
    beta, whole, median, sigma, longest = LONG[kind]
    wl, ap, ad = long_prompts(n_inst, 250, beta, whole, median, sigma, longest)
    ap[::3] = np.minimum(ap[::3], 400)
    route_and_compare(wl, ap, ad, batches=2)
    few = np.minimum(ap, 300)
    few[10::100] = longest
    route_and_compare(wl, few, ad, batches=2)


@pytest.mark.parametrize("n_inst,kind,limit", [(50, "peaks far beyond the threshold", 0.2), (100, "peaks far beyond the threshold", 0.2),
                                               (200, "peaks far beyond the threshold", 0.3), (600, "peaks far beyond the threshold", 0.3),
                                               (100, "half of the prompts beyond exact keys", 0.15), (2000, "large penalty", 0.2)])
def test_batches_that_do_not_fit_exact_keys_are_not_decided_one_by_one_on_all_rows(n_inst, kind, limit):
    """Two thirds of the limit or less; with exact keys (the arrivals that do not fit, or all rows that count as far, outside the loop) well above it."""
    assert share_of_the_scanning_time(*long_prompts(n_inst, 2048, *LONG[kind])) < limit


@pytest.mark.parametrize("n_inst", [257, 300, 1100, 4200])
@pytest.mark.parametrize("n_arr", [1, 4, 5, 9])
@pytest.mark.parametrize("beta", [1.0, 0.75])
def test_a_few_arrivals_on_many_instances(n_inst, n_arr, beta):
    """Both sides of the line up to which no list is built; several batches, short arrivals among them."""
    wl = W.make_random(71, n_inst, 40, 12 * n_inst, 0, max_prompt=300, max_output=60, beta=beta)
    rng = np.random.default_rng(n_arr)
    ap = rng.integers(0, 300, 3 * n_arr).astype(np.int32)
    ad = np.where(rng.random(3 * n_arr) < 0.3, rng.integers(1, 8, 3 * n_arr), rng.integers(8, 60, 3 * n_arr)).astype(np.int32)
    wl.max_requests = 12 * n_inst + 3 * n_arr
    route_and_compare(wl, ap, ad, batches=3)


# the smallest list service, a whole number of passes of the list block and one more, both sides of the line between lists of 128 and of
# 256 rows (and between lists of all rows and of the near ones)
@pytest.mark.parametrize("n_inst", [257, 512, 513, 1024, 1025, 2049])
@pytest.mark.parametrize("beta,t_mem", [(1.0, 0.8), (0.75, 0.8), (0.3, 0.81237)])
@pytest.mark.parametrize("skew", [False, True])
def test_many_lists_in_one_batch(n_inst, beta, t_mem, skew):
    h, n = 40, 24 * n_inst
    wl = W.make_random(72, n_inst, h, n, 0, max_prompt=400, max_output=h, beta=beta)
    wl.t_mem = t_mem
    rng = np.random.default_rng(n_inst)
    if skew:
        wl.instance[:] = np.minimum(n_inst * rng.random(n) ** 3, n_inst - 1).astype(np.int32)
    n_arr = 2200
    ap = np.where(rng.random(n_arr) < 0.02, rng.integers(3000, 6000, n_arr), rng.integers(1, 400, n_arr)).astype(np.int32)
    ad = np.where(rng.random(n_arr) < 0.02, 1, rng.integers(1, 2 * h, n_arr)).astype(np.int32)
    wl.max_requests = n + n_arr
    route_and_compare(wl, ap, ad)


def test_long_prompts_on_thousands_of_rows_find_their_rows_in_the_list():
    """4,096 rows with a window of 100 steps and a deep backlog, prompts to four times the mean: arrivals with prompts beyond the longest one that lists had
    rows for took two lists and a look at all rows each (0.18 of the scanning kernel's time; 0.07 where lists have rows for the longest prompt)."""
    wl = W.make_config(3)
    ap, ad = (dev(x) for x in wl.ticks[0])
    n = len(wl.prompt) + len(ap)
    st = DeviceState(wl.n_instances, 100, wl.capacity_tokens, n + 8192, wl.t_mem, wl.beta, device="cuda:0")
    st.load_requests(wl.prompt, wl.generated, wl.predicted, wl.instance)
    st.make_ring(wl.horizon)
    st.ring_window()
    choice, _ = st.route_batch(ap, ad)
    st.ring_fold(ap, ad, choice)
    queued = st.queued_p.clone()
    best = {}
    for path in (B.ROUTE_AUTO, B.ROUTE_SCAN) * 3:
        st.select_router(path)
        st.ring_window()
        st.n_requests.fill_(n)
        st.queued_p.copy_(queued)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        st.route_batch(ap[:8192], ad[:8192])
        t1.record()
        torch.cuda.synchronize()
        best[path] = min(best.get(path, 1e9), t0.elapsed_time(t1))
    assert st.status() == B.PRE_OK
    st.close()
    assert best[B.ROUTE_AUTO] < 0.11 * best[B.ROUTE_SCAN]


# the line up to which no list is built: two arrivals, and four where all folding warps look at the rows
@pytest.mark.parametrize("n_inst", [257, 2048, 2049])
@pytest.mark.parametrize("n_arr", [2, 3, 4, 5])
@pytest.mark.parametrize("beta", [1.0, 0.75])
def test_arrivals_on_both_sides_of_the_line_for_lists(n_inst, n_arr, beta):
    wl = W.make_random(73, n_inst, 70, 6 * n_inst, 0, max_prompt=300, max_output=90, beta=beta)
    rng = np.random.default_rng(n_inst + n_arr)
    ap, ad = rng.integers(0, 300, 2 * n_arr).astype(np.int32), rng.integers(1, 90, 2 * n_arr).astype(np.int32)
    wl.max_requests = 6 * n_inst + 2 * n_arr
    route_and_compare(wl, ap, ad, batches=2)
