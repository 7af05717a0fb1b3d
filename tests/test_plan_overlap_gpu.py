"""Plans on both sides of the line between overlapped and plain launches."""
import pytest
import torch

import paper_2106_07136_gb300 as bd
import synth
from gpu_helpers import dev, host, same_map

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(120, 160, 1)] * 2, [(120, 160, 3), (121, 161, 1)],
                                   [(120, 160, 4)] * 2, [(240, 320, 1)] * 2, [(240, 321, 1)] * 2,
                                   [(120, 160, 1)] * 3])
def test_plan_groups_are_the_device_batches(sizes):
    """Every group's maps, run after run on refilled images, are the device entry's bit for bit."""
    p = bd.default_params(coarsest_scale=3, gamma=0.5)
    frames = []
    for k in range(2):
        frame = []
        for i, (h, w, count) in enumerate(sizes):
            ps = [synth.make_cfg2(seed=synth.stereo.pair_seed(k, 10 * i + j), h=h, w=w)
                  for j in range(count)]
            frame.append([torch.stack([dev(getattr(q, v), torch.uint8) for q in ps])
                          for v in ("left", "right")])
        frames.append(frame)
    m = bd.Matcher()
    refs = [[host(m.match(l, r, p)) for l, r in frame] for frame in frames]
    groups = [(l.clone(), r.clone(), torch.empty(l.shape, device="cuda")) for l, r in frames[0]]
    plan = bd.Plan(groups, p, autotune=False)
    for frame, ref in list(zip(frames, refs)) * 10:
        for (l, r, _), (lf, rf) in zip(groups, frame):
            l.copy_(lf)
            r.copy_(rf)
        plan.run()
        for (_, _, out), want in zip(groups, ref):
            assert same_map(host(out), want)
    plan.close()
    m.close()
