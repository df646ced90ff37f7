"""Rollouts of networks of different sizes from several host threads at once.
Networks with the same window share a kernel, whose shared memory limit belongs
to the device, not to the call: no call may lower it under another one."""
import threading

import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32,T", [(False, 10), (True, 17)])  # pipelined, persistent kernel
def test_rollouts_of_two_sizes_side_by_side(fp32, T):
    errors, results = [], {}
    start = threading.Barrier(2)

    def work(name, I, H, L, O):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                g = torch.Generator(device="cuda").manual_seed(H)
                net = R.LSTM(I, H, L, O, T, max_batch=2, fp32_weights=fp32)
                net.set_params((torch.rand(net.P, generator=g, device="cuda") * 2 - 1) / H ** 0.5)
                X = torch.randn(2, T, I, generator=g, device="cuda")
                first = net.rollout(X, I - O, 4)
                torch.cuda.current_stream().synchronize()
                start.wait()
                for _ in range(400):
                    out = net.rollout(X, I - O, 4)
                torch.cuda.current_stream().synchronize()
                results[name] = (torch.equal(out, first), net.status())
        except Exception as e:  # noqa: BLE001 - reported below, in the test's thread
            errors.append((name, e))
            start.abort()

    threads = [threading.Thread(target=work, args=a) for a in (("large", 54, 192, 2, 50), ("small", 6, 16, 1, 4))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert results == {"large": (True, R.RPOD_OK), "small": (True, R.RPOD_OK)}
