"""What a network's calls share: buffers across streams, shapes, captures and failures."""
import threading
import time

import numpy as np
import pytest
import torch

import paper_2106_07136_gb300 as bd
from gpu_helpers import dev
from paper_2106_07136_gb300 import _lib

pytestmark = pytest.mark.gpu


def net_batch(seed, count, h, w):
    rng = np.random.default_rng(seed)
    return [dev(rng.uniform(0, hi, (count, h, w)).astype(np.float32)) for hi in (255, 255, 4)]


@pytest.mark.parametrize("shape", [(1, 15, 20), (8, 30, 40), (48, 60, 80)])
def test_forward_beside_gradient(shape):
    """Forward passes on one stream beside gradients on another, of one network: each is what it
    gives alone (the loss to the order of its 32-bit sums), and no wait of a grid barrier runs out."""
    L, R, label = net_batch(1, *shape)
    net = bd.ProposalNet(bd.net_init_weights(seed=6))
    ref, (ref_loss, ref_g) = net.forward(L, R), net.gradient(L, R, label)
    torch.cuda.synchronize()
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    grads, passes, wrong = [], 0, 0

    def train():
        for _ in range(40):
            grads.append(net.gradient(L, R, label, stream=sb))

    t = threading.Thread(target=train)
    t.start()
    with torch.cuda.stream(sa):
        while passes == 0 or t.is_alive():
            outs = [net.forward(L, R, stream=sa) for _ in range(8)]
            passes += len(outs)
            wrong += sum(not torch.equal(o, ref) for o in outs)
    t.join()
    torch.cuda.synchronize()
    net.status()
    assert len(grads) == 40 and wrong == 0
    for loss, g in grads:
        assert np.array_equal(g, ref_g) and abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    net.close()


@pytest.fixture
def net_variant(request):
    old = bd.get_net_variant()
    bd.set_net_variant(request.param)
    yield request.param
    bd.set_net_variant(old)


@pytest.mark.parametrize("net_variant", [0, 1, 2], indirect=True)
def test_a_gradient_whose_wait_ran_out_is_not_a_number(net_variant):
    """The call's word for failed waits, set from the host where a kernel would set it: loss and
    gradient are NaN, a training step leaves the weights, the next calls are as always."""
    L, R, label = net_batch(2, 3, 30, 40)
    net = bd.ProposalNet(bd.net_init_weights(seed=6))
    w0 = net.weights()
    ref_loss, ref = net.gradient(L, R, label)

    def reported():
        with pytest.raises(bd.BdisError) as e:
            net.status()
        assert e.value.status == _lib.BDIS_E_TIMEOUT
        net.status()

    net.inject_timeout()
    loss, g = net.gradient(L, R, label)
    assert np.isnan(loss) and np.isnan(g).all()
    reported()
    net.inject_timeout()
    assert np.isnan(net.train_step(L, R, label, 1e-3))
    reported()
    assert np.array_equal(net.weights(), w0)
    loss, g = net.gradient(L, R, label)
    assert np.array_equal(g, ref) and abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    assert abs(net.train_step(L, R, label, 1e-3) - ref_loss) <= 1e-5 * abs(ref_loss)
    w1 = net.weights()
    assert np.isfinite(w1).all() and not np.array_equal(w1, w0)
    net.status()
    net.close()


@pytest.mark.parametrize("others", [[(2, 9, 12)], [(2, 9, 12), (8, 40, 50), (1, 61, 37), (2, 9, 12)]])
def test_a_captured_forward_pass_outlives_other_shapes(others):
    """Replays of a captured forward pass after eager calls of smaller and larger shapes (and the
    captured one's) through the same network: the eager pass bit for bit."""
    net = bd.ProposalNet(bd.net_init_weights(seed=6))
    L, R, _ = net_batch(3, 4, 30, 40)
    ref = net.forward(L, R)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        out = net.forward(L, R)
    for i, shape in enumerate(others):
        Lo, Ro, _ = net_batch(4 + i, *shape)
        fresh = bd.ProposalNet(bd.net_init_weights(seed=6))
        for _ in range(2):
            o = net.forward(Lo, Ro)
            assert torch.equal(o, fresh.forward(Lo, Ro))
            out.zero_()
            graph.replay()
            assert torch.equal(out, ref)
        fresh.close()
        assert torch.equal(net.forward(L, R), ref)
    torch.cuda.synchronize()
    net.status()
    net.close()


@pytest.mark.parametrize("net_variant", [0, 2], indirect=True)
@pytest.mark.parametrize("shape", [(1, 2, 3), (3, 31, 41), (2, 9, 300)])
def test_two_gradient_buffers_give_the_same_gradient(net_variant, shape):
    """A batch whose layers' gradients cannot all be had holds two at a time: the gradient bit for
    bit, on every call; where those cannot be had either, the failure is reported and the network
    is usable."""
    batch, tiny = net_batch(7, *shape), net_batch(8, 1, 1, 1)
    ref_net, net = (bd.ProposalNet(bd.net_init_weights(seed=6)) for _ in range(2))
    ref_loss, ref = ref_net.gradient(*batch)
    net.gradient(*tiny)  # the sums' buffer, which does not depend on the shape
    try:
        bd.inject_alloc_failures(2)
        with pytest.raises(bd.BdisError) as e:
            net.gradient(*batch)
        assert e.value.status == _lib.BDIS_E_NOMEM
        bd.inject_alloc_failures(1)
        got = [net.gradient(*batch) for _ in range(2)]
    finally:
        bd.inject_alloc_failures(0)
    net.gradient(*tiny)
    got.append(net.gradient(*batch))
    for loss, g in got:
        assert np.array_equal(g, ref) and abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    net.status()
    net.close()
    ref_net.close()


@pytest.mark.parametrize("shape", [(1000, 1, 1), (2000, 5, 5), (700, 40, 2)])
def test_large_batches_of_tiny_images_train_layer_by_layer(shape):
    """The default variant takes the launches per layer there, as variant 2 does: its gradient bit
    for bit; a small batch of the same images does not (within the order of 32-bit sums)."""
    batch = net_batch(9, *shape)
    few = [t[:8].contiguous() for t in batch]
    net = bd.ProposalNet(bd.net_init_weights(seed=6))
    old = bd.get_net_variant()
    try:
        bd.set_net_variant(2)
        ref, ref_few = net.gradient(*batch)[1], net.gradient(*few)[1]
        bd.set_net_variant(1)
        g, g_few = net.gradient(*batch)[1], net.gradient(*few)[1]
    finally:
        bd.set_net_variant(old)
    net.status()
    net.close()
    assert np.array_equal(g, ref)
    assert np.linalg.norm(g_few - ref_few) <= 1e-5 * np.linalg.norm(ref_few)


def test_a_call_costs_the_host_the_same_for_tall_images():
    """Enqueueing a forward pass: the band heights of images of 240 rows are chosen in little more
    time than those of one row (the least of many calls, so that nothing else of the host counts)."""
    net = bd.ProposalNet(bd.net_init_weights(seed=6))

    def least(shape):
        L, R, _ = net_batch(10, *shape)
        best = np.inf
        for _ in range(300):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            net.forward(L, R)
            best = min(best, time.perf_counter() - t0)
        return best

    short, tall = least((1, 1, 135)), least((1, 240, 135))
    net.close()
    assert tall <= 1.5 * short, (short, tall)
