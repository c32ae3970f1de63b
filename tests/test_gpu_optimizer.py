"""Probe position optimizer (Sec. 5) on the GPU against the FP64 oracle: the
room scene, whose grid buries probes in its boxes, with 5 iterations.  The
optimizer picks rays by their hit distances (closest / farthest), so a probe
whose two best candidates lie within FP32 rounding of each other may move
differently; those probes are counted (a handful at most) and masked."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import REL, patched, rel_err, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2009_10796_gb300 as pkg
    pkg.load()
    return pkg


@pytest.fixture(scope="module")
def case():
    sc = synth.room_scene()
    L = synth.room_lights()
    desc = synth.room_volume(optimizer_iters=5, offset_limit=0.45, hysteresis_irr=0.5, hysteresis_vis=0.5)
    h = oracle.SceneHandle(sc)
    st, irr, dist = oracle.new_state(desc)
    off = oracle.new_offsets(desc)
    for f in (0, 1):
        oracle.update(h, L, desc, f, st, irr, dist, offsets=off)
    return sc, L, desc, st, irr, dist, off


def test_optimizer_offsets_states_and_texels(g, case):
    sc, L, desc, st, irr, dist, off = case
    S = g.Scene.from_arrays(sc)
    V = g.Volume(desc)
    for f in (0, 1):
        V.update(S, L, f)
    torch.cuda.synchronize()
    V.poll_status()
    go = V.offsets().cpu().numpy().astype(np.float64)
    moved = np.any(off != 0, axis=1)
    diff = np.abs(go - off).max(1)
    bad = diff > 1e-4
    print(f"[optimizer] probes {len(off)}, moved {int(moved.sum())}, offsets differing {int(bad.sum())}, "
          f"max diff on the rest {diff[~bad].max():.2e}")
    assert moved.sum() > 0.05 * len(off)              # the room buries and crowds many probes
    assert bad.sum() <= max(3, int(0.01 * len(off)))
    lim = 0.45 * np.asarray(desc.spacing)
    assert np.all(np.abs(go) <= lim * (1 + 1e-6))
    gs = V.states().cpu().numpy()
    assert np.array_equal(gs[~bad], st[~bad])
    gi = V.irr_atlas().cpu().numpy()
    gd = V.dist_atlas().cpu().numpy()
    ei = rel_err(gi, irr).max(-1)[~bad]
    ed = rel_err(gd, dist).max(-1)[~bad]
    print(f"[optimizer] texels: irr max {ei.max():.2e}, dist max {ed.max():.2e}")
    assert ei.max() <= REL and ed.max() <= REL
    # end to end, with the probes the two sides moved differently (listed
    # above) taken from the GPU (offset, state, tiles); and the query kernel
    # alone against the oracle's query of the GPU's own atlas, states and offsets
    pos, nrm, cam = synth.room_queries()
    st_p = np.where(bad, gs, st).astype(np.uint8)
    off_p = np.ascontiguousarray(np.where(bad[:, None], go, off))
    E_ref = oracle.query(desc, st_p, patched(irr, gi, np.broadcast_to(bad[:, None, None], gi.shape[:3])),
                         patched(dist, gd, np.broadcast_to(bad[:, None, None], gd.shape[:3])), pos, nrm, cam,
                         offsets=off_p)
    E = V.query(to_dev(pos), to_dev(nrm), cam).cpu().numpy()
    e = rel_err(E, E_ref).max(-1)
    E_own = oracle.query(desc, gs, gi.astype(np.float64), gd.astype(np.float64), pos, nrm, cam,
                         offsets=np.ascontiguousarray(go))
    e_own = rel_err(E, E_own).max(-1)
    print(f"[optimizer] query: max {e.max():.2e} ({int(bad.sum())} listed probes from the GPU); against the "
          f"GPU's own atlas max {e_own.max():.2e}")
    assert e.max() <= REL and e_own.max() <= REL


@pytest.mark.parametrize("rays", [7, 31, 33])
def test_optimizer_ragged_batches(g, rays):
    """Ray counts that leave a batch of 32 rays partly empty (the only one, or the last of two): the
    offsets that the oracle's optimizer gives, up to the few probes of the full test."""
    sc = synth.room_scene()
    desc = synth.room_volume(optimizer_iters=3, rays_per_probe=rays)
    off = oracle.optimize(oracle.SceneHandle(sc), desc, 0, np.arange(desc.n_probes), oracle.new_offsets(desc))
    V = g.Volume(desc)
    V.update(g.Scene.from_arrays(sc), synth.room_lights(), 0)
    bad = np.abs(V.offsets().cpu().numpy() - off).max(1) > 1e-4
    assert np.any(off != 0, axis=1).sum() > 0.05 * len(off)
    assert bad.sum() <= max(3, int(0.01 * len(off)))


def test_optimizer_off_matches_plain_update(g):
    """optimizer_iters = 0 keeps every probe on its grid point."""
    sc = synth.room_scene(n_boxes=6)
    desc = synth.room_volume()
    S = g.Scene.from_arrays(sc)
    V = g.Volume(desc)
    V.update(S, synth.room_lights(), 0)
    assert torch.count_nonzero(V.offsets()) == 0


def test_optimizer_rejected_where_unsupported(g):
    desc = synth.room_volume(optimizer_iters=5)
    with pytest.raises(g.DDGIError):
        g.Cascade([desc])
    with pytest.raises(g.DDGIError):
        g.Volume(synth.room_volume(optimizer_iters=17))
    with pytest.raises(g.DDGIError):
        g.Volume(synth.room_volume(optimizer_iters=5, offset_limit=0.5))
