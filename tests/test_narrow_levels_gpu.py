"""Levels exactly a patch wide, and one column wider: every sample base but 0 (or 0 and 1) leaves
columns outside the image, so the valid set follows the start and changes with the updates."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2106_07136_gb300 as bd
import synth
from attribution import FLAG_DIVERGED
from gpu_helpers import (DROP, DSTAR_ATOL, assert_explained, decision_margins, dev, host,
                         oracle_unstable)
from paper_2106_07136_gb300 import build as cuda_build

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def variants_reset():
    old = bd.get_search_variant(), bd.get_search_tiling()
    yield
    bd.set_search_variant(old[0])
    bd.set_search_tiling(old[1])


def narrow_level(orc, ps, w, h, kw, spread, seed):
    """Oracle planes of a textured strip whose right view is moved by up to 2 px, a start map within
    `spread` px of the shift (whole and fractional), and the oracle's search of it."""
    rng = np.random.default_rng(seed)
    rows = np.arange(h)[:, None]
    x = np.arange(w, dtype=np.float64)[None, :]
    amp, ph = rng.uniform(15, 30, (h, 4)), rng.uniform(0, 6.28, (h, 4))
    freq = rng.uniform(0.25, 0.9, 4)
    shift = 1.0 + np.sin(rows / 9.0)

    def view(at):
        return 120 + sum(amp[:, i:i + 1] * np.sin(freq[i] * at + ph[:, i:i + 1]) for i in range(4))

    op = orc.OracleParams.make(patch_size=ps, overlap=0.75, gamma=0.25, **kw)
    o = dict(L=view(x).astype(np.float32).astype(np.float64),
             R=view(x + shift).astype(np.float32).astype(np.float64))
    o["G"] = orc.sobel_x(o["L"]).astype(np.float32).astype(np.float64)
    ch = (h + 1) // 2
    c = (np.sin(np.arange(ch) / 4.5) + 1 + rng.uniform(-spread, spread, ch)) / 2
    c[::5] = np.round(c[::5])
    o["coarse"] = np.repeat(c.astype(np.float32).astype(np.float64)[:, None], (w + 1) // 2, 1)
    o.update(orc.search_level(o["L"], o["R"], o["G"], o["coarse"], op))
    return o, op


LAYOUTS = [(1, False), (1, True), (2, False), (2, True), (4, False), (4, True)]


def check_against_oracle(orc, ps, wider, kw):
    """Every patch whose oracle result float32 rounding does not move, in all lane layouts: the
    oracle's D*, its reason to drop the patch (DIS: whether it left its range) and, away from a
    whole base, its valid pixels."""
    o, op = narrow_level(orc, ps, ps + wider, 161, kw, 4.0, ps + wider)
    unstable = oracle_unstable(orc, o, op)
    saddle, div, edge = decision_margins(o, ps)
    assert unstable.mean() < 0.1 and (np.abs(o["u_init"]) > 1).mean() > 0.3
    mask = FLAG_DIVERGED if op.fusion else DROP
    sure = ~unstable & (saddle > 1e-4) & (div > 1e-3) & (edge > 1e-3)
    gp = bd.default_params(patch_size=ps, overlap=0.75, gamma=0.25, **kw)
    args = (dev(o["L"]), bd.pack_right(dev(o["R"])), dev(o["G"]), dev(o["coarse"]), gp)
    for variant, tiled in LAYOUTS:
        bd.set_search_variant(variant)
        bd.set_search_tiling(tiled)
        g = {k: host(v)[0] for k, v in bd.search_level(*args).items()}
        np.testing.assert_allclose(g["d_star"][~unstable], o["d_star"][~unstable], atol=DSTAR_ATOL)
        np.testing.assert_array_equal((g["flags"][sure] & mask) != 0, (o["flags"][sure] & mask) != 0)
        np.testing.assert_array_equal(g["n_valid"][sure], o["n_valid"][sure])


@pytest.mark.parametrize("ps", [8, 12, 16])
@pytest.mark.parametrize("wider", [0, 1])
@pytest.mark.parametrize("fusion", [0, 1])
def test_first_update_follows_the_start(orc, ps, wider, fusion):
    """One update from starts of a few pixels either way."""
    check_against_oracle(orc, ps, wider, dict(iterations=1, fusion=fusion))


@pytest.mark.parametrize("ps", [8, 12, 16])
@pytest.mark.parametrize("wider", [0, 1])
@pytest.mark.parametrize("kw", [dict(fusion=0), dict(fusion=1), dict(normalize=0)])
def test_later_updates_follow_the_base(orc, ps, wider, kw):
    """The whole search: each base that an update reaches has its own valid set."""
    check_against_oracle(orc, ps, wider, dict(iterations=12, **kw))


def seeded_frames(w):
    """Two frames of pairs whose coarsest level (of 4) is 8 columns at widths 113 to 128, and the
    disparity of the frame before them."""
    pairs = [synth.make_cfg2(seed=synth.stereo.pair_seed(6, i), h=160, w=w) for i in range(2)]
    prev = np.stack([p.disp for p in pairs]).astype(np.float32)
    return np.stack([p.left for p in pairs]), np.stack([p.right for p in pairs]), prev


NARROW_KW = dict(patch_size=8, overlap=0.75, iterations=12, coarsest_scale=4, finest_scale=0,
                 gamma=0.5)


@pytest.mark.parametrize("w", [113, 128])
def test_warm_start_on_a_coarsest_level_of_one_patch(orc, w):
    L, R, prev = seeded_frames(w)
    gp, op = bd.default_params(**NARROW_KW), orc.OracleParams.make(**NARROW_KW)
    m = bd.Matcher()
    out = host(m.match_warm(dev(L, torch.uint8), dev(R, torch.uint8), dev(prev), gp))
    m.close()
    for i in range(2):
        assert_explained(orc, out[i], L[i], R[i], gp, op, f"{w} wide, frame {i}", budget=False,
                         prev=prev[i])


CHECKED = """
import sys
import numpy as np
sys.path[:0] = sys.argv[2:]
import paper_2106_07136_gb300 as bd
import oracle
import test_narrow_levels_gpu as t
assert bd.checked_build()
out = t.narrow_outputs(oracle)
out["__sites__"] = np.array([bd.check_status()], dtype=np.int64)
np.savez(sys.argv[1], **out)
"""


def narrow_outputs(orc):
    out = {}
    L, R, prev = seeded_frames(128)
    gp = bd.default_params(**NARROW_KW)
    m = bd.Matcher()
    net = bd.ProposalNet(bd.net_init_weights(seed=5))
    for variant, tiled in LAYOUTS:
        bd.set_search_variant(variant)
        bd.set_search_tiling(tiled)
        key = f"{variant} {tiled}"
        Ld, Rd = dev(L, torch.uint8), dev(R, torch.uint8)
        out["warm " + key] = host(m.match_warm(Ld, Rd, dev(prev), gp))
        out["learned " + key] = host(m.match_learned(net, Ld, Rd, gp, fallback=True))
        for ps in (8, 12, 16):
            for wider in (0, 1):
                o, _ = narrow_level(orc, ps, ps + wider, 97, dict(iterations=12), 12.0, ps)
                p = bd.default_params(patch_size=ps, overlap=0.75, gamma=0.25)
                g = bd.search_level(dev(o["L"]), bd.pack_right(dev(o["R"])), dev(o["G"]),
                                    dev(o["coarse"]), p)
                out.update({f"{ps}+{wider} {k} {key}": host(v) for k, v in g.items()})
    net.close()
    m.close()
    return out


def checked_outputs(script, tmp_path):
    """The arrays that `script` saves in a process that loads the bounds-checked build."""
    lib = cuda_build.build(checked=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    (tmp_path / "child.py").write_text(script)
    res = tmp_path / "out.npz"
    r = subprocess.run([sys.executable, str(tmp_path / "child.py"), str(res), root,
                        os.path.join(root, "tests")], env=dict(os.environ, BDIS_LIBRARY=lib),
                       cwd=root, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return dict(np.load(res))


def test_checked_build_catches_nothing(orc, tmp_path):
    """Starts up to 12 px either way: no access of the bounds-checked build is out of bounds, and
    every output is the normal build's bit for bit."""
    got = checked_outputs(CHECKED, tmp_path)
    assert int(got.pop("__sites__")[0]) == 0
    ref = narrow_outputs(orc)
    assert set(got) == set(ref)
    for k in ref:
        assert np.array_equal(got[k], ref[k], equal_nan=ref[k].dtype.kind == "f"), k


TILE = """
import sys
import numpy as np
sys.path[:0] = sys.argv[2:]
import paper_2106_07136_gb300 as bd
import test_narrow_levels_gpu as t
assert bd.checked_build()
out = t.full_tile_outputs()
out["__sites__"] = np.array([bd.check_status()], dtype=np.int64)
np.savez(sys.argv[1], **out)
"""


def full_tile_level(span):
    """Patches of 12 columns, 6 apart, one row of them: two neighbours that share a warp of the
    one-column-per-lane layout start `span` px apart, so that the columns their ranges reach are
    47 + span, and each takes one step of -11.5 px, nearly its whole range, inside the image."""
    ps, w, first, start = 12, 204, 12, -30.0  # patch indices first and first + 1
    x = np.arange(w, dtype=np.float64)
    L = np.broadcast_to(2 * x, (ps, w))
    G = np.full((ps, w), 2.0)
    mid = 6 * first - start + 12 + span / 2  # between the two patches' samples
    R = np.where(x < mid, 2 * (x + start) - 23, 2 * (x + start - span) - 23)
    coarse = np.zeros((ps // 2, w // 2))
    for i, u in ((first, start), (first + 1, start - span)):
        coarse[:, 3 * i + 2:3 * i + 4] = u / 2  # patch i's centre is at 3 i + 2.75
    kw = dict(patch_size=ps, overlap=0.5, iterations=1, normalize=0, gamma=0.25)
    return L, np.broadcast_to(R, (ps, w)), G, coarse, kw, first


SPANS = [46, 47, 48, 49]  # 48 fills the tile's 96 columns; 49 is read from global memory


def full_tile_outputs():
    out = {}
    for span in SPANS:
        L, R, G, coarse, kw, _ = full_tile_level(span)
        for tiled in (False, True):
            bd.set_search_variant(1)
            bd.set_search_tiling(tiled)
            g = bd.search_level(dev(L), bd.pack_right(dev(R)), dev(G), dev(coarse),
                                bd.default_params(**kw))
            out.update({f"{span} {tiled} {k}": host(v) for k, v in g.items()})
    return out


def test_lanes_past_the_patch_stay_in_a_full_tile(tmp_path):
    """Patch 12, one column per lane: four lanes of each group have no column. On a tile whose
    columns are all used, the bounds-checked build finds no read past it; outputs as untiled."""
    got = checked_outputs(TILE, tmp_path)
    assert int(got.pop("__sites__")[0]) == 0
    ref = full_tile_outputs()
    for span in SPANS:
        first = full_tile_level(span)[-1]
        d, u = ref[f"{span} True d_star"][0, 0], ref[f"{span} True u_init"][0, 0]
        np.testing.assert_allclose((d - u)[first:first + 2], -11.5, atol=1e-3)
        np.testing.assert_allclose(u[first] - u[first + 1], span, atol=1e-3)
    for k in ref:
        assert np.array_equal(got[k], ref[k], equal_nan=ref[k].dtype.kind == "f"), k
        assert np.array_equal(ref[k], ref[k.replace("True", "False")],
                              equal_nan=ref[k].dtype.kind == "f"), k
