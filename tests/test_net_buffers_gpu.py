"""What a network's calls share: buffers across streams, shapes, captures and failures."""
import threading

import numpy as np
import pytest
import torch

import paper_2106_07136_gb300 as bd
from gpu_helpers import dev

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
        while t.is_alive():
            outs = [net.forward(L, R, stream=sa) for _ in range(8)]
            passes += len(outs)
            wrong += sum(not torch.equal(o, ref) for o in outs)
    t.join()
    torch.cuda.synchronize()
    net.status()
    assert len(grads) == 40 and passes > 0 and wrong == 0
    for loss, g in grads:
        assert np.array_equal(g, ref_g) and abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    net.close()
