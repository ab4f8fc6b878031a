"""Entropy plans of several orders called from several host threads, a stream
each: every call succeeds and gives what it gives alone. The orders ask for
different amounts of shared memory of the same kernel (256 on clusters of 5
CTAs, 512 on clusters of 2 and 1024 on clusters of 4), which is a limit of the
kernel on the device and not of one launch. States with a NaN make a call
short (the reduction ends at once, the entropy is NaN), so that the threads
launch as often as they can.
"""
import threading

import numpy as np
import pytest
import torch

import paper_2203_09353_gb300 as bg

pytestmark = pytest.mark.gpu

# walkers, spins, split, calls
CASES = [(4, 7, 6, 3000), (4, 9, 8, 3000), (60, 10, 9, 3000), (30, 11, 10, 1000)]


def test_orders_side_by_side(gpu):
    rng = np.random.default_rng(3)
    runs = []
    for walkers, spins, split, calls in CASES:
        x = rng.standard_normal((walkers, 2, 1 << spins))
        x = x[:, 0] + 1j * x[:, 1]
        finite = torch.from_numpy(x.copy()).cuda()
        x[:, 0] = np.nan
        states = torch.from_numpy(x).cuda()
        plan = bg.entropy_plan(walkers, spins, split)
        alone = torch.zeros(walkers, dtype=torch.float64, device="cuda")
        bg.batched_entropy(plan, finite, alone)
        out = torch.zeros_like(alone)
        runs.append((plan, states, finite, alone, out, calls, torch.cuda.Stream()))
    torch.cuda.synchronize()
    failed = []

    def work(plan, states, finite, alone, out, calls, stream):
        try:
            for _ in range(calls):
                bg.batched_entropy(plan, states, out, stream=stream)
            stream.synchronize()
            assert torch.isnan(out).all()
            bg.batched_entropy(plan, finite, out, stream=stream)
            stream.synchronize()
            assert torch.equal(out, alone)
        except Exception as e:  # noqa: BLE001 (reported by the test's own thread)
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=r) for r in runs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    bg.check_device_errors()
