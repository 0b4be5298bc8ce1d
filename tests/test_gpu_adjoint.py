"""GPU adjoint of the alignment objective against the fp64 oracle and central
differences, and its torch.autograd wrapper."""
import numpy as np
import pytest

import oracle
from paper_2207_03936_gb300 import synth
from tests.test_oracle_alignment import central_differences, truth_tracks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the library stores hit_sigma as fp32; the oracle gets the same value
SIGMA = float(np.float32(0.012))


@pytest.fixture(scope="module")
def setup():
    from paper_2207_03936_gb300 import sbt
    ev = synth.make_events(5, 40, workers=1)
    ho, th = truth_tracks(ev)
    h = sbt.sbt_create(ev.module_z, sbt.default_config(hit_sigma=SIGMA))
    d = {k: torch.from_numpy(v).cuda() for k, v in
         dict(x=ev.x, y=ev.y, z=ev.z, m=ev.module, ho=ho, th=th).items()}
    yield sbt, h, ev, ho, th, d
    h.close()


def test_adjoint_matches_oracle_gradient(setup):
    sbt, h, ev, ho, th, d = setup
    rng = np.random.default_rng(8)
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    c, g = sbt.sbt_fit_adjoint(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"],
                               torch.from_numpy(align).cuda())
    torch.cuda.synchronize()
    v, go = oracle.align_chi2(ev.x, ev.y, ev.z, ev.module, ho, th, ev.module_z, align, SIGMA)
    assert abs(float(c.item()) - v) <= 1e-12 * v
    g = g.cpu().numpy()
    scale = np.abs(go).max()
    assert (np.abs(g - go) <= 1e-9 * np.maximum(np.abs(go), 1e-3 * scale)).all()


def test_adjoint_against_central_differences(setup):
    # 12 events keep the objective small enough (~3e6) for fp64 differences
    # to resolve every gradient entry to better than 1e-6
    sbt, h, _, _, _, _ = setup
    ev = synth.make_events(5, 12, workers=1)
    ho, th = truth_tracks(ev)
    d = [torch.from_numpy(a).cuda() for a in (ev.x, ev.y, ev.z, ev.module, ho, th)]
    rng = np.random.default_rng(9)
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    _, g = sbt.sbt_fit_adjoint(h, *d, torch.from_numpy(align).cuda())
    g = g.cpu().numpy()
    fd = central_differences(
        lambda a: oracle.align_chi2(ev.x, ev.y, ev.z, ev.module, ho, th, ev.module_z, a, SIGMA,
                                    False)[0], align)
    scale = np.abs(fd).max()
    assert (np.abs(g - fd) <= 1e-6 * np.maximum(np.abs(fd), 1e-3 * scale)).all()


def test_adjoint_is_bitwise_reproducible(setup):
    sbt, h, ev, ho, th, d = setup
    a = torch.zeros(52, 6, dtype=torch.float64, device="cuda")
    c1, g1 = sbt.sbt_fit_adjoint(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"], a)
    c2, g2 = sbt.sbt_fit_adjoint(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"], a)
    assert torch.equal(c1, c2) and torch.equal(g1, g2)


def test_autograd_function(setup):
    sbt, h, ev, ho, th, d = setup
    a = torch.zeros(52, 6, dtype=torch.float64, device="cuda", requires_grad=True)
    loss = sbt.alignment_chi2(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"], a)
    (2.0 * loss).backward()
    _, g = sbt.sbt_fit_adjoint(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"], a.detach())
    assert torch.allclose(a.grad, 2.0 * g, rtol=0, atol=0)
    # a small step along -grad lowers the objective by about eta * |grad|^2
    with torch.no_grad():
        f0 = float(loss.detach())
        eta = 1e-4 * f0 / float((g * g).sum())
        l2 = sbt.alignment_chi2(h, d["x"], d["y"], d["z"], d["m"], d["ho"], d["th"], a - eta * g)
    assert f0 - float(l2) > 0.5e-4 * f0


def test_adjoint_on_reconstructed_tracks(setup):
    sbt, h, ev, ho, th, d = setup
    out = sbt.sbt_reconstruct_batched(h, d["x"], d["y"], d["z"], d["m"],
                                      torch.from_numpy(ev.event_offsets).cuda())
    r = out.compact()
    a = np.zeros((52, 6))
    c, g = sbt.sbt_fit_adjoint(h, d["x"], d["y"], d["z"], d["m"],
                               torch.from_numpy(r["hit_offsets"]).cuda(),
                               torch.from_numpy(r["track_hits"]).cuda(), torch.from_numpy(a).cuda())
    v, go = oracle.align_chi2(ev.x, ev.y, ev.z, ev.module, r["hit_offsets"], r["track_hits"],
                              ev.module_z, a, SIGMA)
    assert abs(float(c.item()) - v) <= 1e-12 * v
    # the fp64 objective at zero alignment equals the sum of the fp32 fits
    assert abs(v - float(r["chi2"].astype(np.float64).sum())) <= 1e-3 * v


def test_adjoint_on_long_repeated_and_invalid_tracks(setup):
    # tracks of 104 hits (two per module), a repeated module, and tracks
    # without a line fit or with indices out of range (skipped and counted):
    # the same value, gradient and count as the oracle's
    sbt, h, _, _, _, _ = setup
    from tests.hand_events import MZ
    from tests.test_oracle_alignment import _odd_tracks
    x, y, z, m, good = _odd_tracks()
    x, y, z = (np.append(a, np.float32(a[0])) for a in (x, y, z))
    m = np.append(m, np.int32(52))
    bad = [np.array([11]), np.array([], np.int64), np.array([5, 5 + 52]), np.array([1, 2, 105]),
           np.array([58, 59, 104, 61])]
    allt = [good[0], bad[0], good[1], bad[1], bad[2], good[2], bad[3], bad[4]] * 40
    th = np.concatenate(allt).astype(np.int32)
    ho = np.concatenate([[0], np.cumsum([len(t) for t in allt])]).astype(np.int32)
    rng = np.random.default_rng(21)
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    d = [torch.from_numpy(a).cuda() for a in (x, y, z, m, ho, th)]
    c, g, sk = sbt.sbt_fit_adjoint(h, *d, torch.from_numpy(align).cuda(), with_skipped=True)
    torch.cuda.synchronize()
    v, go, so = oracle.align_chi2(x, y, z, m, ho, th, MZ, align, SIGMA, count_skipped=True)
    assert int(sk.item()) == so == 5 * 40
    assert abs(float(c.item()) - v) <= 1e-12 * v
    g = g.cpu().numpy()
    scale = np.abs(go).max()
    assert (np.abs(g - go) <= 1e-9 * np.maximum(np.abs(go), 1e-3 * scale)).all()
    # reproducible to the bit with the repeated-module path taken
    c2, g2, _ = sbt.sbt_fit_adjoint(h, *d, torch.from_numpy(align).cuda(), with_skipped=True)
    assert torch.equal(c.cpu(), c2.cpu()) and np.array_equal(g, g2.cpu().numpy())


@pytest.mark.parametrize("lengths", [[3], [2, 1, 0], [64], [65, 64, 2, 63], [20, 24, 17, 33], [200, 3, 5]],
                         ids=lambda v: "-".join(map(str, v)))
@pytest.mark.parametrize("n_tracks", [1, 31, 129, 2000])
def test_adjoint_tiles(setup, n_tracks, lengths):
    """Tiles of tracks by hits and by number (1536 hits, 128 tracks: full,
    exceeded, one short), tracks at and above the longest of a tile, tracks
    without a fit in between, fewer tracks than blocks; random hits, so that
    modules repeat within tracks."""
    sbt, h, ev, _, _, d = setup
    rng = np.random.default_rng([n_tracks, *lengths])
    n = np.resize(np.array(lengths), n_tracks)
    ho = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    th = rng.integers(0, ev.n_hits, int(ho[-1])).astype(np.int32)
    if n_tracks > 100 and len(th) > 500:
        th[len(th) // 2] = ev.n_hits      # one track with an index out of range
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    args = [d["x"], d["y"], d["z"], d["m"], torch.from_numpy(ho).cuda(), torch.from_numpy(th).cuda(),
            torch.from_numpy(align).cuda()]
    c, g, sk = sbt.sbt_fit_adjoint(h, *args, with_skipped=True)
    c2, g2 = sbt.sbt_fit_adjoint(h, *args)
    v, go, so = oracle.align_chi2(ev.x, ev.y, ev.z, ev.module, ho, th, ev.module_z, align, SIGMA,
                                  count_skipped=True)
    assert int(sk.item()) == so
    # residuals of centimetres: the fp64 sums agree to a few thousand roundings;
    # residuals that vanish (two hits) are left with about ten roundings of
    # coordinates up to 750 mm, delta = 1e-12 mm a hit, at lever arms up to 42 mm
    delta, hits = 1e-12, len(th)
    assert abs(float(c.item()) - v) <= 1e-12 * v + hits * (delta / SIGMA) ** 2
    assert np.abs(g.cpu().numpy() - go).max() <= 1e-11 * np.abs(go).max() + hits * 2 * delta / SIGMA ** 2 * 42
    assert torch.equal(c, c2) and torch.equal(g, g2)


@pytest.mark.parametrize("per_module", [1, 2, 8, 32, 100])
def test_adjoint_long_tracks_that_share_modules(setup, per_module):
    """Tracks above 64 hits whose hits share modules in every multiplicity of a
    round of 32 lanes (one hit a lane and module up to all 32 on one module)."""
    sbt, h, ev, _, _, d = setup
    rng = np.random.default_rng(per_module)
    by_module = [np.flatnonzero(ev.module == m) for m in range(52)]
    tracks = [np.concatenate([rng.choice(by_module[m], per_module) for m in rng.permutation(52)])[:300]
              for _ in range(40)]
    tracks = [np.resize(t, 66 + 7 * k) for k, t in enumerate(tracks)]
    ho = np.concatenate([[0], np.cumsum([len(t) for t in tracks])]).astype(np.int32)
    th = np.concatenate(tracks).astype(np.int32)
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    args = [d["x"], d["y"], d["z"], d["m"], torch.from_numpy(ho).cuda(), torch.from_numpy(th).cuda(),
            torch.from_numpy(align).cuda()]
    c, g = sbt.sbt_fit_adjoint(h, *args)
    c2, g2 = sbt.sbt_fit_adjoint(h, *args)
    v, go = oracle.align_chi2(ev.x, ev.y, ev.z, ev.module, ho, th, ev.module_z, align, SIGMA)
    # fp64 sums in another order; residuals of centimetres
    assert abs(float(c.item()) - v) <= 1e-12 * v
    assert np.abs(g.cpu().numpy() - go).max() <= 1e-11 * np.abs(go).max()
    assert torch.equal(c, c2) and torch.equal(g, g2)


@pytest.mark.parametrize("lengths", [[3], [2, 1, 0], [65, 64, 2, 63], [20, 24, 17, 33], [200, 3, 5], [160]],
                         ids=lambda v: "-".join(map(str, v)))
@pytest.mark.parametrize("n_tracks", [0, 1, 31, 129, 2000])
def test_adjoint_value_only(setup, n_tracks, lengths):
    """A call without a gradient leaves out forces, torques and their order by
    module: the value and the skipped count stay those of the full call, bit
    for bit, with invalid tracks among them."""
    sbt, h, ev, _, _, d = setup
    rng = np.random.default_rng([n_tracks, *lengths])
    ho = np.concatenate([[0], np.cumsum(np.resize(np.array(lengths), n_tracks))]).astype(np.int32)
    th = rng.integers(0, ev.n_hits, int(ho[-1])).astype(np.int32)
    if n_tracks > 100 and len(th) > 500:
        th[len(th) // 2] = ev.n_hits
    align = np.concatenate([rng.normal(0, 0.005, (52, 3)), rng.normal(0, 5e-5, (52, 3))], 1)
    args = [d["x"], d["y"], d["z"], d["m"], torch.from_numpy(ho).cuda(), torch.from_numpy(th).cuda(),
            torch.from_numpy(align).cuda()]
    c, g, sk = sbt.sbt_fit_adjoint(h, *args, with_skipped=True)
    c2, none, sk2 = sbt.sbt_fit_adjoint(h, *args, want_grad=False, with_skipped=True)
    assert none is None and g.shape == (52, 6)
    assert torch.equal(c, c2) and torch.equal(sk, sk2)


@pytest.mark.parametrize("value", [3e38, np.inf, np.nan], ids=str)
def test_adjoint_beyond_fp32_sums(setup, value):
    """Positions whose fp32 sum overflows keep the fp64 result; infinities and
    NaN reach the same entries as in the oracle."""
    sbt, h, ev, ho, th, d = setup
    x = ev.x.copy()
    t = int(np.argmax(np.diff(ho)))
    mine = th[ho[t]:ho[t + 1]]
    if np.isfinite(value):
        x[mine] = value * np.linspace(0.5, 1.0, len(mine), dtype=np.float32) ** 2
    else:
        x[mine[1]] = value
    align = np.zeros((52, 6))
    c, g = sbt.sbt_fit_adjoint(h, torch.from_numpy(x).cuda(), d["y"], d["z"], d["m"], d["ho"], d["th"],
                               torch.from_numpy(align).cuda())
    with np.errstate(invalid="ignore"):
        v, go = oracle.align_chi2(x, ev.y, ev.z, ev.module, ho, th, ev.module_z, align, SIGMA)
    g = g.cpu().numpy()
    if np.isfinite(value):
        assert np.isfinite(go).all() and abs(float(c.item()) - v) <= 1e-12 * v
        # per parameter: n roundings at the scale of its largest entry
        assert (np.abs(g - go).max(0) <= 1e-12 * np.abs(go).max(0)).all()
    else:
        assert np.isnan(v) and np.isnan(float(c.item()))
        assert np.isnan(go).any() and (np.isnan(g) == np.isnan(go)).all()
