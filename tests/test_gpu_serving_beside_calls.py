"""Served jobs and blocking calls side by side on one device: launch limits, memory, waiting.  Nothing is faulted."""
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
