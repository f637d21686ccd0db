"""Served jobs and blocking calls side by side on one device: launch limits, memory, waiting.  Nothing is faulted."""
import ctypes
import threading
import time

import pytest

import paper_2512_01055_gb300 as tc
from tests.test_gpu_fp64_tensor import _random

pytestmark = pytest.mark.gpu


def _args(d):
    return [d[n] for n in ("eps", "t1", "t2", "ovvv", "ovoo", "ovov")]


@pytest.mark.parametrize("prec,slices", [(tc.TC_FP64, 0), (tc.TC_SPLIT_BF16, 3)])
def test_launches_of_one_kernel_with_different_shared_memory(prec, slices):
    """Jobs of v = 20 and v = 40, served and in blocking calls of several contexts, run one kernel instance with
    different amounts of shared memory from many host threads: none may change the limit another launches under."""
    import torch
    data = {v: _random(2, v, v) for v in (20, 40)}
    torch.cuda.synchronize()
    bad, end = [], time.monotonic() + 4.0

    def loop(v, served):
        ctx = tc.tc_init(0)
        try:
            while time.monotonic() < end:
                if served:
                    t = tc.tc_submit(ctx, 2, v, *_args(data[v]), prec=prec, slices=slices, device_inputs=True)
                    code, _ = tc.tc_wait(ctx, t, 60000)
                    if code != tc.TC_OK:
                        bad.append(("served", v, code))
                else:
                    tc.tc_energy_dev(ctx, 2, v, *_args(data[v]), prec=prec, slices=slices,
                                     stream=torch.cuda.Stream())
        except tc.TcError as e:
            bad.append(("call", v, str(e)))
        finally:
            tc.tc_finalize(ctx)

    ths = [threading.Thread(target=loop, args=a) for a in [(20, False), (40, False)] * 3 + [(20, True), (40, True)]]
    for th in ths:
        th.start()
    for th in ths:
        th.join()
    assert not bad, (len(bad), bad[:2])


def _used(free):
    import torch
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


SLACK = 48 << 20        # small buffers, 2 MB allocation granularity, kernels loaded on first use


def _trim():
    """Give the device's memory pool, which keeps served jobs' memory for reuse, back to the device."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool = ctypes.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0


def _warm():
    """Every kernel and the caching allocator's blocks in place, so that only contexts' buffers change the free memory."""
    d = _random(3, 24, 9)
    ctx = tc.tc_init(0)
    for prec in (tc.TC_FP64, tc.TC_SPLIT_BF16):
        tc.tc_energy_dev(ctx, 3, 24, *_args(d), prec=prec, slices=4)
        code, _ = tc.tc_wait(ctx, tc.tc_submit(ctx, 3, 24, *_args(d), prec=prec, slices=4, device_inputs=True), 60000)
        assert code == tc.TC_OK
    tc.tc_finalize(ctx)
    _trim()


def test_residue_images_and_the_buffers_of_earlier_calls():
    """Split images of most of the budget, then an FP64 call, then a split call again: the context never holds more
    than the budget, and each call runs on its own path."""
    import torch
    small, large = _random(4, 64, 64), _random(10, 128, 65)
    need = tc.tc_workspace_bytes(10, 128, tc.TC_SPLIT_BF16, 4)
    budget = need + (32 << 20)                        # the images of o=4 v=64 take about 115 MB
    _warm()
    free = torch.cuda.mem_get_info()[0]
    ctx = tc.tc_init(0, hbm_budget_bytes=budget)
    try:
        for _ in range(2):
            tc.tc_energy_dev(ctx, 10, 128, *_args(large), prec=tc.TC_SPLIT_BF16, slices=4)
            print(f"budget {budget >> 20} MB, used after the split call {_used(free) >> 20} MB")
            assert _used(free) <= budget + SLACK
            r = tc.tc_energy_dev(ctx, 4, 64, *_args(small), prec=tc.TC_FP64)
            assert r.prep_seconds > 0.0 and 64 << 20 < _used(free) <= budget + SLACK      # residues, kept
    finally:
        tc.tc_finalize(ctx)


def test_residue_images_beside_the_context_s_own_inputs():
    """A host call's inputs are in use: with no room for the images beside them the DMMA kernel runs."""
    d = _random(4, 64, 64)
    host = [x.cpu().numpy() for x in _args(d)]
    inputs = sum(x.nbytes for x in host)
    for extra, dmma in ((64 << 20, True), (256 << 20, False)):
        ctx = tc.tc_init(0, hbm_budget_bytes=inputs + extra)
        try:
            r = tc.tc_energy(ctx, 4, 64, *host, prec=tc.TC_FP64)
            assert (r.prep_seconds == 0.0) == dmma
        finally:
            tc.tc_finalize(ctx)


def test_kept_residue_images_give_way_to_served_jobs_in_the_budget():
    """Images kept after a blocking FP64 call, then a served job of nearly the whole budget."""
    import torch
    small, large = _random(4, 64, 64), _random(10, 128, 65)
    budget = tc.tc_workspace_bytes(10, 128, tc.TC_SPLIT_BF16, 4) + (32 << 20)
    _warm()
    free = torch.cuda.mem_get_info()[0]
    ctx = tc.tc_init(0, hbm_budget_bytes=budget)
    try:
        r = tc.tc_energy_dev(ctx, 4, 64, *_args(small), prec=tc.TC_FP64)
        assert r.prep_seconds > 0.0 and _used(free) > 64 << 20
        t = tc.tc_submit(ctx, 10, 128, *_args(large), prec=tc.TC_SPLIT_BF16, slices=4, device_inputs=True)
        code, _ = tc.tc_wait(ctx, t, 60000)
        assert code == tc.TC_OK
        print(f"budget {budget >> 20} MB, used {_used(free) >> 20} MB")       # the pool keeps the job's memory
        assert _used(free) <= budget + SLACK
    finally:
        tc.tc_finalize(ctx)


@pytest.mark.parametrize("prec,slices", [(tc.TC_SPLIT_BF16, 4), (tc.TC_FP64, 0)])
def test_kept_residue_images_give_way_to_served_jobs_on_a_full_device(prec, slices):
    """The device has less room than the budget: the job that fits once the images are given back runs.  (FP64 with
    its own images of the same size: it takes the room rather than the DMMA kernel.)"""
    import torch
    large = _random(10, 128, 65)
    ctx = tc.tc_init(0, hbm_budget_bytes=8 << 30)
    fill = None
    try:
        ref = tc.tc_energy_dev(ctx, 10, 128, *_args(large), prec=tc.TC_FP64)      # about 1.3 GB of images, kept
        assert ref.prep_seconds > 0.0
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        _trim()
        fill = torch.empty(torch.cuda.mem_get_info()[0] - (768 << 20), dtype=torch.uint8, device="cuda")
        t = tc.tc_submit(ctx, 10, 128, *_args(large), prec=prec, slices=slices, device_inputs=True)
        code, r = tc.tc_wait(ctx, t, 60000)
        assert code == tc.TC_OK
        if prec == tc.TC_FP64:
            assert r.e_t == ref.e_t
    finally:
        del fill
        tc.tc_finalize(ctx)


def test_first_job_starts_while_clients_keep_handing_in():
    """Twelve clients hand in small host jobs without a pause for 1.5 s (most are refused: the queue is short), so a
    batch is always about to grow: the first job starts after a quarter of an iteration, 0.25 s, not when the clients
    are done."""
    d = _random(3, 120, 66)
    host = [x.cpu().numpy() for x in _args(d)]
    ctx = tc.tc_init(0, iteration_ms=1000, max_inflight=4, max_queue=8)
    tickets, lock = [], threading.Lock()

    def client(end):
        while time.monotonic() < end:
            try:
                t = tc.tc_submit(ctx, 3, 120, *host, prec=tc.TC_SPLIT_BF16, slices=3)
            except tc.TcError as e:
                assert e.status == tc.TC_EBUSY
                continue
            with lock:
                tickets.append(t)

    try:
        code, _ = tc.tc_wait(ctx, tc.tc_submit(ctx, 3, 120, *host, prec=tc.TC_SPLIT_BF16, slices=3), 60000)
        assert code == tc.TC_OK                                         # threads, kernels and pool are in place
        ths = [threading.Thread(target=client, args=(time.monotonic() + 1.5,)) for _ in range(12)]
        for th in ths:
            th.start()
        for th in ths:
            th.join()
        done = {}
        for t in tickets:
            code, done[t] = tc.tc_wait(ctx, t, 120000)
            assert code == tc.TC_OK
        first = done[min(done)].queue_seconds
        print(f"{len(tickets)} jobs taken, the first started after {first:.3f} s")
        assert first < 0.75
    finally:
        tc.tc_finalize(ctx)
