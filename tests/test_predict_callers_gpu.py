"""UNet.predict among other users of the process: it runs the forward pass on the caller's stream and nothing else."""
import threading

import pytest
import torch

from paper_2409_01076_gb300 import unet as U

pytestmark = pytest.mark.gpu


def image(seed, n=1, side=64):
    return torch.rand(n, side, side, 3, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


def test_other_threads_may_wait_for_the_device():
    """A recording in progress would make their synchronisation an error."""
    x = image(1)
    U.UNet(base=32).predict(x)
    stop, errors = threading.Event(), []

    def waiter():
        try:
            while not stop.is_set():
                torch.cuda.synchronize()
        except Exception as e:          # noqa: BLE001
            errors.append(e)

    th = threading.Thread(target=waiter)
    th.start()
    try:
        for k in range(20):
            net = U.UNet(base=32, seed=k)
            want = net.forward(x, None)
            for _ in range(4):
                assert torch.equal(net.predict(x), want)
    finally:
        stop.set()
        th.join()
    assert not errors, errors[0]


def test_inference_mode_then_not():
    net, x = U.UNet(base=32, seed=2), image(2)
    with torch.inference_mode():
        inside = [net.predict(x).cpu() for _ in range(3)]
    for _ in range(3):
        assert torch.equal(net.predict(x).cpu(), inside[0])


def test_replaced_parameters_are_read():
    """Biases and the head's weights are looked up at every call."""
    net, x = U.UNet(base=32, seed=3), image(3)
    for _ in range(3):
        before = net.predict(x)
    net.params["head.w"] = 2.0 * net.params["head.w"]
    net.params["head.b"] = 2.0 * net.params["head.b"]
    assert torch.equal(net.predict(x), 2.0 * before)
    net.params["dec1b.b"] = net.params["dec1b.b"] + 1.0
    assert not torch.equal(net.predict(x), 2.0 * before)


def test_predictions_keep_no_memory():
    net, x = U.UNet(base=32, seed=4), image(4, 4, 256)
    net.predict(x)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    for _ in range(4):
        net.predict(x)
    torch.cuda.empty_cache()
    held = torch.cuda.memory_reserved()
    assert torch.cuda.memory_allocated() == before and held <= before + (64 << 20)
