"""The blocking host entry's chunks."""
import numpy as np
import pytest
import torch

import paper_2106_07136_gb300 as bd

pytestmark = pytest.mark.gpu

KW = dict(iterations=3, coarsest_scale=2, gamma=0.25)


def pairs(w, h, count):
    rng = np.random.default_rng(count)
    tile = rng.integers(0, 256, (3, h, w + 8), dtype=np.uint8)
    idx = rng.integers(0, 3, count)
    return [torch.from_numpy(np.ascontiguousarray(tile[idx][:, :, o:o + w])) for o in (5, 8)]


def same(a, b):
    return torch.equal(a.view(torch.int32), b.view(torch.int32))


@pytest.mark.parametrize("w,h,count", [(640, 480, 2), (640, 480, 7), (640, 480, 13), (640, 480, 49),
                                       (1601, 1203, 41)])
def test_a_workspace_that_cannot_be_had_takes_smaller_chunks(w, h, count):
    left, right = pairs(w, h, count)
    p = bd.default_params(**KW)
    m = bd.Matcher("cuda:0")
    ref = m.match_host(left.pin_memory(), right.pin_memory(), p)
    whole = m.workspace_bytes
    m.close()
    m = bd.Matcher("cuda:0")
    bd.inject_alloc_failures(1)
    try:
        out = m.match_host(left.pin_memory(), right.pin_memory(), p)
        assert m.workspace_bytes <= 0.8 * whole
        assert same(out, ref)
        bd.inject_alloc_failures(2)
        fresh = bd.Matcher("cuda:0")
        with pytest.raises(bd.BdisError) as e:
            fresh.match_host(left, right, p)
        assert e.value.status == bd._lib.BDIS_E_NOMEM
    finally:
        bd.inject_alloc_failures(0)
    assert same(fresh.match_host(left.pin_memory(), right.pin_memory(), p), ref)
    fresh.close()
    m.close()


@pytest.mark.parametrize("kw,longest", [(dict(KW, overlap=0.25, finest_scale=1), 20),
                                        (dict(KW, overlap=0.5), 20), (dict(KW, iterations=12), 48)])
def test_fast_settings_take_chunks_of_equal_length(kw, longest):
    """64 pairs: settings whose match takes no longer than a few copies run in chunks of at most 20
    (seen by the workspace: pyramid, patches and two sets of images of the longest chunk), the
    default's kind in one of 48 between two short ones; the device entry's maps either way."""
    left, right = pairs(640, 480, 64)
    p = bd.default_params(**kw)
    m, r = bd.Matcher("cuda:0"), bd.Matcher("cuda:0")
    out = m.match_host(left.pin_memory(), right.pin_memory(), p)
    r.reserve(640, 480, longest, p)
    images = 2 * 640 * 480 * longest * 6
    assert r.workspace_bytes < m.workspace_bytes <= r.workspace_bytes + images + (1 << 16)
    assert same(out, r.match(left.cuda(), right.cuda(), p).cpu())
    m.close()
    r.close()


@pytest.mark.parametrize("kw", [KW, dict(KW, overlap=0.25, finest_scale=1)])
@pytest.mark.parametrize("w,h,count", [(640, 480, 13), (640, 480, 49), (1601, 1203, 41)])
def test_pageable_memory_through_the_chunks(kw, w, h, count):
    """Graded and even splits from and to memory that is not pinned, twice through one handle: the
    device entry's maps."""
    left, right = pairs(w, h, count)
    p = bd.default_params(**kw)
    m = bd.Matcher("cuda:0")
    outs = [m.match_host(left, right, p, torch.empty(count, h, w)) for _ in range(2)]
    ref = m.match(left.cuda(), right.cuda(), p).cpu()
    m.close()
    for out in outs:
        assert not out.is_pinned() and same(out, ref)
