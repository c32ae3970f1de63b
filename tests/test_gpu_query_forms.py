"""The query's specialised forms (storage format, gamma, probe offsets fixed at compile time)
and the general one against the FP64 oracle on the same stored values, and the grouping of the
query's adjoint, on seeded atlases whose depth variance is a fixed share of the depth squared
(so no Chebyshev weight is near a cancellation), and the forms once more where it nearly cancels."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import REL, fp32_texel_spread, rel_err, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2009_10796_gb300 as pkg
    pkg.load()
    torch.cuda.set_device(0)
    return pkg


FORMS = {   # irradiance format, distance format, gamma, offsets
    "fp32": (0, 0, 5.0, False), "half": (1, 1, 5.0, False), "rgb9e5": (2, 0, 5.0, False),
    "moved": (0, 0, 5.0, True), "gamma1": (0, 0, 1.0, False), "half_fp32": (1, 0, 5.0, False),
    "gamma2": (0, 0, 2.0, False), "moved_half": (1, 1, 5.0, True),
    "half_gamma1": (1, 1, 1.0, False), "half_gamma2.2": (1, 1, 2.2, False), "rgb9e5_gamma2.2": (2, 0, 2.2, False),
}


def _volume(g, form, irr_n=5, dist_n=7, counts=(3, 4, 2), cancelling=False):
    fi, fd, gamma, moved = FORMS[form]
    desc = synth.VolumeDesc(origin=(0.5, -0.25, 1.0), spacing=(1.0, 1.25, 1.5), counts=counts, rays_per_probe=37,
                            irr_n=irr_n, dist_n=dist_n, gamma=gamma, optimizer_iters=int(moved), seed=5)
    V = g.Volume(desc, irr_format=fi, dist_format=fd)
    rng, P, N, M = synth.Rng(11), desc.n_probes, irr_n + 2, dist_n + 2
    irr = rng.uniform(P * N * N * 3, 0.05, 1.0).reshape(P, N, N, 3)
    mean = rng.uniform(P * M * M, 0.3, 2.5).reshape(P, M, M)
    dist = np.stack([mean, 1.3 * mean * mean], -1)
    if cancelling:      # one depth a probe, its variance 1e-5 to 1e-3 of its square
        mean = np.broadcast_to(rng.uniform(P, 0.3, 1.5)[:, None, None], mean.shape)
        dist = np.stack([mean, mean * mean * (1.0 + 10.0 ** rng.uniform(P, -5.0, -3.0)[:, None, None])], -1)
    if fi == 2:
        q = np.floor(irr * 256).astype(np.int64)                     # exponent 16: steps of 2^-8
        V.set_buffer(0, torch.tensor((q[..., 0] | (q[..., 1] << 9) | (q[..., 2] << 18) | (16 << 27)).astype(np.uint32).view(np.int32), device="cuda"))
        irr = q / 256.0
    else:
        dt = torch.float16 if fi == 1 else torch.float32
        t = torch.zeros((P, N, N, 4), dtype=dt, device="cuda")
        t[..., :3] = to_dev(irr).to(dt)
        V.set_buffer(0, t)
        irr = t[..., :3].double().cpu().numpy()
    d = to_dev(dist).to(torch.float16 if fd == 1 else torch.float32)
    V.set_buffer(1, d)
    states = np.full(P, 4, dtype=np.uint8)
    states[1::7] = 2                                                 # some asleep: cages with missing corners
    V.set_buffer(2, torch.tensor(states, device="cuda"))
    off = None
    if moved:
        off = np.zeros((P, 4))
        off[:, :3] = synth.f32(rng.uniform(3 * P, -0.3, 0.3).reshape(P, 3))
        V.set_buffer(3, to_dev(off))
        off = np.ascontiguousarray(off[:, :3])                       # as the oracle takes them
    return desc, V, states, irr, d.double().cpu().numpy(), off


def _points(n, seed):
    rng = synth.Rng(seed)
    pos = synth.f32(rng.uniform(3 * n, -1.0, 5.0).reshape(n, 3))      # inside the grid and around it
    nrm = rng.unit_vectors(n)
    nrm[5::11] = 0.0                                                  # background pixels
    return pos, nrm, np.array([1.0, 2.0, 0.5])


@pytest.mark.parametrize("n", [1, 257])
@pytest.mark.parametrize("form", list(FORMS))
def test_query_forms_match_oracle(g, form, n):
    desc, V, st, irr, dist, off = _volume(g, form)
    pos, nrm, cam = _points(n, 21)
    E = V.query(to_dev(pos), to_dev(nrm), cam).cpu().numpy()
    assert rel_err(E, oracle.query(desc, st, irr, dist, pos, nrm, cam, offsets=off)).max() <= REL
    dirs = synth.Rng(23).unit_vectors(n)
    M = V.query_glossy(to_dev(pos), to_dev(nrm), to_dev(dirs)).cpu().numpy()
    assert rel_err(M, oracle.query_glossy(desc, st, irr, dist, pos, nrm, dirs, offsets=off)).max() <= REL


def _arranged(kind):
    """Points by the groups of equal cage and footprint that a warp of them has."""
    if kind == "one":
        return _points(1, 31)
    pos, nrm, cam = _points(333, 37)
    if kind == "same":                                                # whole warps of one group, and a tail
        pos[:] = pos[0] + synth.f32(synth.Rng(41).uniform(333 * 3, 0, 1e-3).reshape(-1, 3))
        nrm[:] = nrm[0]
    elif kind == "few":                                               # three groups, interleaved
        pos, nrm = pos[np.arange(333) % 3], nrm[np.arange(333) % 3]
    return pos, nrm, cam                                              # "scattered": a group a point


@pytest.mark.parametrize("fold", [False, True])
@pytest.mark.parametrize("kind", ["one", "same", "few", "scattered"])
@pytest.mark.parametrize("form", ["fp32", "half", "rgb9e5", "moved", "gamma1", "gamma2"])
def test_texel_gradient_groups(g, form, kind, fold):
    """All contributions of one sign (dE > 0), so the sums meet the parity tolerance texel by texel."""
    desc, V, st, irr, dist, off = _volume(g, form)
    pos, nrm, cam = _arranged(kind)
    dE = synth.f32(synth.Rng(43).uniform(3 * len(pos), 0.5, 1.5).reshape(-1, 3))
    G = V.query_backward(to_dev(pos), to_dev(nrm), cam, to_dev(dE), fold_borders=fold).cpu().numpy()
    R = oracle.query_texel_grad(desc, st, irr, dist, pos, nrm, cam, dE, fold=fold, offsets=off)
    assert rel_err(G, R).max() <= REL


@pytest.mark.parametrize("form", ["fp32", "half", "rgb9e5", "moved", "gamma1", "gamma2", "half_fp32", "half_gamma1"])
def test_query_forms_where_the_variance_cancels(g, form):
    """Depths of almost no variance, so that mu2 - mu^2 cancels to a few hundred ulps in every Chebyshev
    weight beyond the mean: each point within the parity tolerance plus twice what the oracle's own
    result moves by when the stored values move by four FP32 ulps (the rounding of the moments' sums
    and of mu^2 is below that)."""
    desc, V, st, irr, dist, off = _volume(g, form, cancelling=True)
    pos, nrm, cam = _points(257, 51)
    keep = np.any(nrm != 0.0, axis=1)
    pos, nrm = pos[keep], nrm[keep]
    if off is not None:
        off = np.zeros_like(off)                                     # the spread's oracle has none
        V.set_buffer(3, to_dev(np.zeros((desc.n_probes, 4))))
    E = V.query(to_dev(pos), to_dev(nrm), cam).cpu().numpy().astype(np.float64)
    ref = oracle.query(desc, st, irr, dist, pos, nrm, cam)
    spread = fp32_texel_spread(desc, st, irr, dist, pos, nrm, np.broadcast_to(cam, pos.shape))
    e = (np.abs(E - ref) / np.maximum(np.abs(ref), 1e-30)).max(-1)
    assert (spread > REL).sum() > 10                                 # the weights do depend on the last bits
    assert (e <= REL + 2.0 * spread).all()


@pytest.mark.parametrize("n", [1, 257])
def test_rgb9e5_gamma1_matches_oracle(g, monkeypatch, n):
    """The one form of point queries that the table above has no row for."""
    monkeypatch.setitem(FORMS, "rgb9e5_gamma1", (2, 0, 1.0, False))
    test_query_forms_match_oracle(g, "rgb9e5_gamma1", n)
