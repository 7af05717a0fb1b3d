"""Kernels chosen by size, type or alignment, at the edges of their ranges,
against a plain restatement that rounds the same way (bit for bit), or the
general kernel they stand in for."""
import numpy as np
import pytest
import torch

import paper_2106_07136_gb300 as bd
from gpu_helpers import dev, host
from oracle import net_oracle as no

pytestmark = pytest.mark.gpu


def _warm_map_f32(p, level):
    """Row-major float32 sums of each block's finite values, as the header states the map."""
    b, h, w = p.shape
    s = 1 << level
    lo = s // 2
    out = np.zeros((b, -(-h // s), -(-w // s)), np.float32)
    for i in range(b):
        for y in range(out.shape[1]):
            for x in range(out.shape[2]):
                v = p[i, max(y * s - lo, 0):y * s + lo, max(x * s - lo, 0):x * s + lo]
                v = v[np.isfinite(v)]
                if v.size:
                    out[i, y, x] = np.add.accumulate(v, dtype=np.float32)[-1] / \
                        np.float32(v.size) / np.float32(s)
    return out


@pytest.mark.parametrize("level,shape", [(1, (5, 7)), (2, (33, 65)), (3, (16, 24)), (3, (61, 301)),
                                         (4, (97, 515)), (5, (120, 160)), (5, (135, 257)),
                                         (6, (200, 333)), (7, (90, 1100)), (9, (70, 90)),
                                         (13, (20, 30)), (14, (20, 30))])
def test_warm_map_is_the_row_major_float32_mean(level, shape):
    rng = np.random.default_rng(level * 1000 + shape[1])
    p = rng.uniform(0.0, 60.0, size=(3, *shape)).astype(np.float32)
    p[rng.random(p.shape) < 0.1] = np.nan
    p[0, :3, :3] = np.inf
    p[1, : shape[0] // 2] = np.nan
    p[2, 1::5, 2::3] = -0.0
    np.testing.assert_array_equal(host(bd.warm_map(dev(p), level)), _warm_map_f32(p, level))


@pytest.mark.parametrize("ps,overlap", [(8, 0.75), (8, 0.5), (6, 0.6), (32, 0.9), (5, 0.0)])
@pytest.mark.parametrize("count,shape", [(1, (33, 61)), (2, (67, 33)), (40, (161, 321))])
def test_dis_densify_geometry(orc, ps, overlap, count, shape):
    """DIS fusion over patch grids of other strides, with weights other than 1, dropped patches
    and D* beyond the image; 5e-4 px as for the other DIS stages, the same unestimated pixels."""
    h, w = shape
    kw = dict(patch_size=ps, overlap=overlap, iterations=4, coarsest_scale=0, finest_scale=0,
              fusion=bd._lib.BDIS_FUSION_DIS)
    gp, op = bd.default_params(**kw), orc.OracleParams.make(**kw)
    _, nx = bd.grid(w, ps, overlap)
    _, ny = bd.grid(h, ps, overlap)
    rng = np.random.default_rng(ps + count)
    d = rng.uniform(-6, 40, (count, ny, nx)).astype(np.float32)
    d[..., ::4] = np.round(d[..., ::4])  # whole samples: the last column is inside
    weight = np.where(rng.random(d.shape) < 0.5, 1.0, rng.uniform(0.1, 2.0, d.shape))
    weight = np.where(rng.random(d.shape) < 0.3, 0.0, weight).astype(np.float32)
    d[weight == 0] = np.nan
    L = rng.uniform(0, 255, (count, h, w)).astype(np.float32)
    R = np.clip(L + rng.normal(0, 2, L.shape), 0, 255).astype(np.float32)
    out = host(bd.densify_level((h, w), gp, dev(d), dev(weight), None, True, dev(L),
                                bd.pack_right(dev(R))))
    for i in {0, count - 1}:
        ref = orc.densify_level((h, w), op, np.nan_to_num(d[i]), weight[i], None, True, L[i], R[i])
        assert np.array_equal(np.isnan(out[i]), np.isnan(ref))
        np.testing.assert_allclose(out[i], ref, atol=5e-4)


@pytest.mark.parametrize("count,h,w", [(8, 1, 1), (2, 2, 129), (4, 33, 5), (2, 9, 300), (16, 31, 41)])
@pytest.mark.parametrize("variant", [1, 2])
def test_weight_gradient_of_a_batch_is_the_mean_of_its_images(count, h, w, variant):
    """Both layouts training runs in. Images smaller than a tile, narrower than a tap, wider than a tile, and tiles that hold
    several images. For a power of two of images every activation and activation gradient of the
    batch is that of the image alone (scaled exactly), so the gradients differ by the order of
    32-bit sums only: 1e-5 of each layer's norm. The gradient is the same every time."""
    rng = np.random.default_rng(w)
    L = rng.uniform(0, 255, (count, h, w)).astype(np.float32)
    R = rng.uniform(0, 255, (count, h, w)).astype(np.float32)
    label = rng.uniform(0, 4, (count, h, w)).astype(np.float32)
    label[rng.random(label.shape) < 0.1] = np.nan
    net = bd.ProposalNet(bd.net_init_weights(seed=w))
    old = bd.get_net_variant()
    try:
        bd.set_net_variant(variant)
        loss, g = net.gradient(dev(L), dev(R), dev(label))
        assert np.array_equal(net.gradient(dev(L), dev(R), dev(label))[1], g)
        each = [net.gradient(dev(L[i]), dev(R[i]), dev(label[i])) for i in range(count)]
        bd.set_net_variant(3 - variant)
        other = net.gradient(dev(L), dev(R), dev(label))[1]
    finally:
        bd.set_net_variant(old)
    net.status()
    net.close()
    assert np.linalg.norm(g - other) <= 1e-5 * np.linalg.norm(other)
    assert abs(loss - np.mean([e[0] for e in each])) <= 1e-5 * loss
    mean = np.mean([e[1].astype(np.float64) for e in each], axis=0)
    off = 0
    for ci, co in no.CHANNELS:
        n = co * 9 * ci + co
        a, b = g[off:off + n], mean[off:off + n]
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b), (ci, co)
        off += n


def _planes(h, w, count, seed):
    rng = np.random.default_rng(seed)
    wide = np.cumsum(rng.normal(0, 12, (count, h, w + 16)), axis=2) % 200 + 20
    shift = rng.integers(0, 6, count)
    left = np.stack([v[:, 8:8 + w] for v in wide])
    right = np.stack([v[:, 8 + k:8 + k + w] for v, k in zip(wide, shift)])
    right = right + rng.normal(0, 1.0, right.shape)
    return bd.prepare_level0(dev(left.astype(np.float32)), dev(right.astype(np.float32)))


@pytest.mark.parametrize("ps", [4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 15, 16])
@pytest.mark.parametrize("kw", [dict(window_samples=7, window_step=0.4),
                                dict(window_samples=1, gamma=0.25),
                                dict(window_samples=15, window_step=0.25, normalize=0),
                                dict(window_samples=5, window_step=1.0, iterations=0),
                                dict(window_samples=3, fusion=bd._lib.BDIS_FUSION_DIS)])
def test_four_lane_search_is_the_one_column_search(ps, kw):
    """Patches of 4 lanes (each taking every fourth column) against one column per lane, every
    output bit for bit, on images a patch wide up to some tens of patches, with flat and
    non-finite regions, from 0 and from a coarse map."""
    gp = bd.default_params(**dict(dict(patch_size=ps, overlap=0.6, iterations=9), **kw))
    old = bd.get_search_variant()
    for i, (h, w, count) in enumerate([(ps, ps, 1), (ps + 3, 2 * ps + 1, 2), (61, 97, 3)]):
        L, R, G = _planes(h, w, count, 100 * ps + i)
        if i == 2:
            L[0, :30, :40] = 90.0
            G[0, :30, :40] = 0.0
            R[1, 20:24, 50:53, 0] = float("nan")
            R[2, 5, 10, 1] = float("inf")
        coarse = torch.rand(count, (h + 1) // 2, (w + 1) // 2, device=L.device) * 4 if i else None
        outs = []
        try:
            for v in (1, 2):
                bd.set_search_variant(v)
                outs.append({k: host(t) for k, t in
                             bd.search_level(L, R, G, coarse, gp).items()})
        finally:
            bd.set_search_variant(old)
        for key in outs[0]:
            if kw.get("fusion") and key == "energies":
                continue  # not written
            a, b = outs[0][key], outs[1][key]
            assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f"), (h, w, key)


@pytest.mark.parametrize("level,mshape,shape", [(0, (5, 7), (5, 7)), (1, (31, 41), (62, 81)),
                                                (1, (1, 1), (2, 2)), (2, (40, 67), (157, 265)),
                                                (3, (9, 130), (70, 1033))])
def test_upsample_is_the_float32_bilinear(level, mshape, shape):
    """Against a restatement with the same float32 operations (products and sums kept apart:
    2e-6 relative for fused ones), missing values included."""
    rng = np.random.default_rng(level + shape[1])
    m = rng.uniform(0, 30, (2, *mshape)).astype(np.float32)
    m[rng.random(m.shape) < 0.15] = np.nan
    m[1, 0, 0] = np.inf
    sc = np.float32(2 ** level)
    fx = np.minimum(np.arange(shape[1], dtype=np.float32) / sc, np.float32(mshape[1] - 1))
    fy = np.minimum(np.arange(shape[0], dtype=np.float32) / sc, np.float32(mshape[0] - 1))
    x0, y0 = np.floor(fx).astype(int), np.floor(fy).astype(int)
    x1, y1 = np.minimum(x0 + 1, mshape[1] - 1), np.minimum(y0 + 1, mshape[0] - 1)
    tx, ty = (fx - x0)[None, :], (fy - y0)[:, None]
    s = np.zeros((2, *shape), np.float32)
    sw = np.zeros((2, *shape), np.float32)
    for wt, yy, xx in (((1 - tx) * (1 - ty), y0, x0), (tx * (1 - ty), y0, x1),
                       ((1 - tx) * ty, y1, x0), (tx * ty, y1, x1)):
        v = m[:, yy][:, :, xx]
        ok = (wt > 0) & np.isfinite(v)
        s += np.where(ok, wt * np.nan_to_num(v, posinf=0), 0).astype(np.float32)
        sw += np.where(ok, wt, 0).astype(np.float32)
    with np.errstate(invalid="ignore"):
        ref = np.where(sw > 0, sc * s / sw, np.nan)
    out = host(bd.upsample(dev(m), level, shape))
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    np.testing.assert_allclose(out, ref, rtol=2e-6)


@pytest.mark.parametrize("w,h,count", [(640, 480, 11), (640, 480, 13), (1601, 1200, 2),
                                       (1280, 960, 9), (640, 480, 49), (1601, 1203, 41)])
def test_host_chunks_are_the_device_batch(w, h, count):
    """Batches that run whole and in 2, 3 and 5 chunks: the device entry's maps, bit for bit."""
    rng = np.random.default_rng(count)
    tile = rng.integers(0, 256, (3, h, w + 8), dtype=np.uint8)
    idx = rng.integers(0, 3, count)
    left = torch.from_numpy(np.ascontiguousarray(tile[idx][:, :, 5:5 + w])).pin_memory()
    right = torch.from_numpy(np.ascontiguousarray(tile[idx][:, :, 8:8 + w])).pin_memory()
    p = bd.default_params(iterations=3, coarsest_scale=2, gamma=0.25)
    m = bd.Matcher("cuda:0")
    out = m.match_host(left, right, p, torch.empty(count, h, w).pin_memory())
    again = m.match_host(left, right, p, torch.empty(count, h, w).pin_memory())
    ref = m.match(left.cuda(), right.cuda(), p).cpu()
    m.close()
    assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    assert torch.equal(again.view(torch.int32), ref.view(torch.int32))


def _net_batch(seed, count, h, w):
    rng = np.random.default_rng(seed)
    return [dev(rng.uniform(0, hi, (count, h, w)).astype(np.float32)) for hi in (255, 255, 4)]


def test_network_buffers_across_shapes():
    """Larger, smaller and differently padded shapes in turn through one network: what a network
    that has seen only that shape gives, bit for bit (the loss to the order of its 32-bit sums).
    A shape whose planar buffers cannot be had takes the other layout: 1e-5 of the norm."""
    weights = bd.net_init_weights(seed=3)
    shapes = [(4, 30, 40), (2, 9, 12), (4, 29, 43), (1, 61, 37), (4, 30, 40), (3, 12, 9)]
    net = bd.ProposalNet(weights)
    for i, shape in enumerate(shapes):
        L, R, label = _net_batch(i, *shape)
        only = bd.ProposalNet(weights)
        assert np.array_equal(host(net.forward(L, R)), host(only.forward(L, R)))
        loss, g = net.gradient(L, R, label)
        ref_loss, ref = only.gradient(L, R, label)
        only.close()
        assert np.array_equal(g, ref) and abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    L, R, label = _net_batch(9, 6, 50, 50)
    bd.inject_alloc_failures(1)
    try:
        loss, g = net.gradient(L, R, label)
    finally:
        bd.inject_alloc_failures(0)
    ref_loss, ref = net.gradient(L, R, label)
    net.status()
    net.close()
    assert np.linalg.norm(g - ref) <= 1e-5 * np.linalg.norm(ref)
    assert abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)


def test_rows_beyond_a_grid_dimension(orc):
    """More rows of blocks than a launch's second dimension holds."""
    h, w, ps = 8 * 65535 + 21, 9, 8
    rng = np.random.default_rng(1)
    m = rng.uniform(0, 30, ((h + 1) // 2, (w + 1) // 2)).astype(np.float32)
    m[::7, 1] = np.nan
    out = host(bd.upsample(dev(m[None]), 1, (h, w)))[0]
    tail = 64  # the last rows alone, from the map's last rows (an even first row)
    first = (h - tail) // 2 * 2
    ref = host(bd.upsample(dev(m[None, first // 2:]), 1, (h - first, w)))[0]
    np.testing.assert_array_equal(out[first:], ref)
    np.testing.assert_array_equal(out[::2, ::2], 2 * m)
    kw = dict(patch_size=ps, overlap=0.0, coarsest_scale=0, finest_scale=0,
              fusion=bd._lib.BDIS_FUSION_DIS)
    ny, nx = bd.grid(h, ps, 0.0)[1], bd.grid(w, ps, 0.0)[1]
    d = rng.uniform(0, 2, (1, ny, nx)).astype(np.float32)
    weight = np.ones_like(d)
    L = rng.uniform(0, 255, (1, h, w)).astype(np.float32)
    out = host(bd.densify_level((h, w), bd.default_params(**kw), dev(d), dev(weight), None, True,
                                dev(L), bd.pack_right(dev(L))))
    ref = orc.densify_level((h, w), orc.OracleParams.make(**kw), d[0], weight[0], None, True,
                            L[0], L[0])
    assert np.array_equal(np.isnan(out[0]), np.isnan(ref))
    np.testing.assert_allclose(out[0], ref, atol=5e-4)


def test_dis_reciprocal_is_the_division():
    """The block route that takes the weight as a reciprocal against the one that divides (one
    weight of each block other than 1), on the pixels that patch does not cover, bit for bit."""
    ps, h, w = 8, 256, 512
    kw = dict(patch_size=ps, overlap=0.5, coarsest_scale=0, finest_scale=0,
              fusion=bd._lib.BDIS_FUSION_DIS)
    ny, nx = bd.grid(h, ps, 0.5)[1], bd.grid(w, ps, 0.5)[1]
    rng = np.random.default_rng(3)
    d = rng.uniform(0, 3, (8, ny, nx)).astype(np.float32)
    L = rng.uniform(0, 255, (8, h, w)).astype(np.float32)
    R = rng.uniform(0, 255, (8, h, w)).astype(np.float32)
    one = np.ones_like(d)
    other, touched = one.copy(), np.zeros((h, w), bool)
    for j in range(0, ny, 2):  # a patch every 8 rows and 32 columns: one in each block at least
        for i in range(1, nx, 8):
            other[:, j, i] = 0.5
            touched[4 * j:4 * j + ps, 4 * i:4 * i + ps] = True
    a, b = (host(bd.densify_level((h, w), bd.default_params(**kw), dev(d), dev(v), None, True,
                                  dev(L), bd.pack_right(dev(R)))) for v in (one, other))
    keep = ~touched
    keep[:, :40] = False  # blocks at the image's left edge test every sample anyway
    assert keep.mean() > 0.5
    np.testing.assert_array_equal(a[:, keep], b[:, keep])


@pytest.mark.parametrize("ps", [8, 16])
@pytest.mark.parametrize("kw", [dict(), dict(overlap=0.5, normalize=0), dict(iterations=0),
                                dict(fusion=bd._lib.BDIS_FUSION_DIS)])
@pytest.mark.parametrize("h,w", [(16, 16), (61, 98), (64, 160)])
def test_paired_loads_and_inner_warps(ps, kw, h, w):
    """The search that reads the left planes in pairs against the same planes on an odd float (read
    one by one), and warps inside the image against the same warps with a patch that starts far
    outside it: every output of every patch with the same start, bit for bit."""
    gp = bd.default_params(**dict(dict(patch_size=ps, iterations=9), **kw))
    L, R, G = _planes(h, w, 3, h + ps)
    L[0, :30, :40] = 90.0
    G[0, :30, :40] = 0.0
    R[1, 10, 9, 0] = float("nan")
    near = torch.rand(3, (h + 1) // 2, (w + 1) // 2, device=L.device) * 2
    far = near.clone()
    far[:, ::6, ::9] = 1.0e4

    def odd(t):
        v = torch.empty(t.numel() + 1, device=t.device)[1:].view(t.shape)
        assert v.data_ptr() % 8 == 4
        return v.copy_(t)

    def run(left, grad, coarse):
        return {k: host(t) for k, t in bd.search_level(left, R, grad, coarse, gp).items()}

    def same(a, b, where):
        for key in a:
            if kw.get("fusion") and key == "energies":
                continue  # not written
            x, y = a[key][where], b[key][where]
            assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f"), key

    a, b = run(L, G, near), run(L, G, far)
    everywhere = np.ones(a["u_init"].shape, bool)
    for coarse, ref in ((near, a), (far, b), (None, run(L, G, None))):
        same(ref, run(odd(L), odd(G), coarse), everywhere)
    same(a, b, a["u_init"] == b["u_init"])
