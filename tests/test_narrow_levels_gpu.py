"""Levels exactly a patch wide, and one column wider: every sample base but 0 (or 0 and 1) leaves
columns outside the image, so the valid set of the first update follows the start."""
import numpy as np
import pytest

import paper_2106_07136_gb300 as bd
from attribution import FLAG_DIVERGED
from gpu_helpers import DROP, DSTAR_ATOL, decision_margins, dev, host, oracle_unstable

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
