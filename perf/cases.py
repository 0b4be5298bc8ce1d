"""The work that users of this library have it do, as cases to be measured.

Events are drawn on the GPU with the recipe of `synth.py` (same planes,
vertices, tracks, kinks, efficiency, smearing and noise), so that a state is
made in a fraction of a second.  Every state owns a handle, its inputs and its
output buffers, as a program that reconstructs a stream of batches does.
Reconstruction is exact by contract (track sets, hit lists and fits are
bitwise those of the plain definition); the alignment adjoint is fp64 sums.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2207_03936_gb300 import sbt, synth

SIGMA = 0.012


def listed():
    return [
        # one average event reconstructed as it arrives (trigger latency)
        dict(name="event", entry="plain", events=1, pv="fixed", pv_mean=8, **_UPGRADE),
        # a handful of quiet events, one vertex each: the smallest real call
        dict(name="quiet_events", entry="plain", events=16, pv="fixed", pv_mean=1, **_QUIET),
        # a bunch of 500 upgrade events per call, the paper's way of running
        dict(name="bunch_500", entry="plain", events=500, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # 100 events inside an application that owns the device's memory
        dict(name="noalloc_100", entry="noalloc", events=100, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # 1000 upgrade events replayed from a graph, launch shape left at its default
        dict(name="batched_1000", entry="batched", events=1000, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # offline reconstruction: a large batch of uneven events on a tuned handle
        dict(name="batched_uneven", entry="batched", tuned=True, events=16000, pv="uniform", pv_mean=10.5, **_UPGRADE),
        # the same kind of batch with fp16 hit storage and the busiest events cut
        dict(name="batched_fp16_cut", entry="batched", tuned=True, events=6000, pv="uniform", pv_mean=10.5,
             **{**_UPGRADE, "fp16": True, "cut": 10000}),
        # module pairs (the real detector's two sides), ~2000 hits an event
        dict(name="batched_pairs", entry="batched", tuned=True, events=6000, pv="poisson", pv_mean=7.6,
             **{**_UPGRADE, "pairs": True}),
        # from pinned host buffers to pinned host results, copies overlapped by chunks
        dict(name="host_13000", entry="host", tuned=True, events=13000, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # events submitted one by one to the serving loop, results polled
        dict(name="serve_256", entry="serve", events=256, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # alignment: one gradient step on a few events through autograd
        dict(name="align_step_60", entry="align_step", events=60, pv="poisson", pv_mean=7.6, **_UPGRADE),
        # alignment: value and gradient over the full sample of 10000 events
        dict(name="align_10000", entry="align", events=10000, pv="poisson", pv_mean=7.6, **_UPGRADE),
    ]


# tracks per vertex, backward tracks, multiple scattering; storage and geometry options
_UPGRADE = dict(tracks=25.0, backward=0.1, kink=0.5e-3, fp16=False, pairs=False, ascending=False, cut=0, k=4)
_QUIET = dict(tracks=30.0, backward=0.0, kink=0.0, fp16=False, pairs=False, ascending=False, cut=0, k=4)

# largest batch of each entry in a draw, in vertices: the hits follow them
_MOST_PV = dict(plain=20000, batched=120000, noalloc=800, host=80000, serve=2000, align=60000, align_step=4000)


def draw(rng):
    entry = rng.choice(["plain", "plain", "batched", "batched", "batched", "noalloc", "host", "serve", "align",
                        "align_step"])
    align = entry.startswith("align")
    pv = rng.choice(["fixed", "poisson", "uniform"])
    pv_mean = rng.choice([1, 2, 3, 5, 8, 12]) if pv == "fixed" else round(rng.uniform(2.0, 10.5), 1)
    most = min(16000.0, _MOST_PV[entry] / pv_mean)
    if entry == "noalloc":
        # most of 524288 hits: 553 a vertex, with room for the spread of the draw
        most = min(most, 400.0 / pv_mean)
    events = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most))))))
    c = dict(entry=entry, events=events, pv=pv, pv_mean=pv_mean, **_UPGRADE)
    c["tracks"] = round(rng.uniform(15.0, 30.0), 1)
    if not align:
        c["fp16"] = rng.random() < 0.25
        c["pairs"] = rng.random() < 0.25
        c["ascending"] = rng.random() < 0.25
        c["k"] = rng.choice([4, 4, 4, 2, 3, 6])
        if rng.random() < 0.2:
            c["cut"] = int(1.3 * pv_mean * 553 * c["tracks"] / 25.0) + 1
        if entry in ("batched", "host"):
            c["tuned"] = rng.random() < 0.5 and events >= 1000
    return c


# --------------------------------------------------------------- events ---


def _planes():
    return torch.tensor(synth.module_z_ascending(), dtype=torch.float32, device="cuda")


def _chunk(case, g, n_ev, zasc, truth):
    """Hits of n_ev events, shuffled inside each event: x, y, z, plane, counts
    and, for truth, the particle of every hit (-1: noise) and their number."""
    cu = dict(device="cuda")
    mean = float(case["pv_mean"])

    def rand(n):
        return torch.rand(n, generator=g, **cu)

    def randn(*n):
        return torch.randn(*n, generator=g, **cu)

    if case["pv"] == "fixed":
        npv = torch.full((n_ev,), int(mean), dtype=torch.int64, **cu)
    elif case["pv"] == "poisson":
        npv = torch.poisson(torch.full((n_ev,), mean, **cu), generator=g).long()
    else:
        npv = torch.randint(1, int(2 * mean - 1) + 1, (n_ev,), generator=g, **cu)
    ev = torch.repeat_interleave(torch.arange(n_ev, **cu), npv)
    n = ev.numel()
    vz, vx, vy = 60.0 * randn(n), 0.03 * randn(n), 0.03 * randn(n)
    nf = torch.poisson(torch.full((n,), float(case["tracks"]), **cu), generator=g).long()
    nb = torch.poisson(torch.full((n,), float(case["tracks"]) * case["backward"], **cu), generator=g).long()
    pv = torch.repeat_interleave(torch.arange(n, **cu), nf + nb)
    t = pv.numel()
    first = torch.repeat_interleave(torch.cumsum(nf + nb, 0) - nf - nb, nf + nb)
    fwd = torch.arange(t, **cu) - first < nf[pv]
    tant = torch.tan(2.0 * torch.atan(torch.exp(-(2.0 + 3.0 * rand(t)))))
    phi = 2.0 * math.pi * rand(t)
    # columns in travel order: ascending planes forward, descending backward
    M = zasc.numel()
    cols = torch.arange(M, **cu)
    k = torch.where(fwd[:, None], cols, M - 1 - cols)
    z = zasc[k]
    u = torch.where(fwd[:, None], z - vz[pv][:, None], vz[pv][:, None] - z)
    near = (u > 0) & (u * tant[:, None] > synth.R_MIN - 3.0 * synth.PITCH * tant[:, None]) & (
        u * tant[:, None] < synth.R_MAX + 3.0 * synth.PITCH * tant[:, None])

    def along(v0, slope):
        p = v0[pv][:, None] + slope[:, None] * u
        if case["kink"] > 0:
            kick = case["kink"] * randn(t, M) * near
            c1, c2 = torch.cumsum(kick, 1) - kick, torch.cumsum(kick * u, 1) - kick * u
            p += u * c1 - c2
        return p

    x, y = along(vx, tant * torch.cos(phi)), along(vy, tant * torch.sin(phi))
    r2 = x * x + y * y
    keep = near & (r2 >= synth.R_MIN ** 2) & (r2 <= synth.R_MAX ** 2)
    keep &= torch.rand(t, M, generator=g, **cu) < 0.98
    x += SIGMA * randn(t, M)
    y += SIGMA * randn(t, M)
    if case["pairs"]:
        keep &= torch.where(k % 2 == 0, x >= 1.0e-3, x <= -1.0e-3)
    part = torch.arange(t, **cu)[:, None].expand(t, M)[keep]
    x, y, z, k = x[keep], y[keep], z[keep], k[keep]
    hev = ev[pv[part]]
    noise = torch.poisson(0.01 * torch.bincount(hev, minlength=n_ev).float(), generator=g).long()
    nev = torch.repeat_interleave(torch.arange(n_ev, **cu), noise)
    m = nev.numel()
    nk = torch.randint(0, M, (m,), generator=g, **cu)
    nr = torch.sqrt(synth.R_MIN ** 2 + (synth.R_MAX ** 2 - synth.R_MIN ** 2) * rand(m))
    na = 2.0 * math.pi * rand(m)
    nx = nr * torch.cos(na)
    if case["pairs"]:
        nx = torch.where(nk % 2 == 0, 1.0, -1.0) * torch.clamp(nx.abs(), min=1.0e-3)
    x, y = torch.cat([x, nx]), torch.cat([y, nr * torch.sin(na)])
    z, k, hev = torch.cat([z, zasc[nk]]), torch.cat([k, nk]), torch.cat([hev, nev])
    key = (hev << 31) | torch.randint(0, 1 << 31, (x.numel(),), generator=g, **cu)
    order = torch.sort(key)[1]
    part = torch.cat([part, torch.full((m,), -1, dtype=torch.int64, **cu)])[order] if truth else None
    return x[order], y[order], z[order], k[order], torch.bincount(hev, minlength=n_ev), part, t


def _events(case, seed, truth=False):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    zasc = _planes()
    M = zasc.numel()
    per = max(1, int(20000 / max(1.0, float(case["pv_mean"]))))
    got, parts, base, total = [], [], 0, 0
    for e0 in range(0, int(case["events"]), per):
        *c, part, t = _chunk(case, g, min(per, int(case["events"]) - e0), zasc, truth)
        got.append(c)
        if truth:
            parts.append(torch.where(part >= 0, part + base, part))
        base += t
        total += c[0].numel()
    x, y, z, k, counts = (torch.cat(v) for v in zip(*got))
    offsets = torch.zeros(counts.numel() + 1, dtype=torch.int32, device="cuda")
    offsets[1:] = torch.cumsum(counts, 0)
    mz, mz2 = synth.module_z_traversal(), None
    if case["pairs"]:
        p = synth.module_z_ascending().reshape(synth.N_PAIRS, 2)[::-1].astype(np.float32)
        mz, mz2 = p[:, 0].copy(), p[:, 1].copy()
        module = synth.N_PAIRS - 1 - k // 2
    else:
        module = M - 1 - k
    if case["ascending"]:
        module = len(mz) - 1 - module
        mz, mz2 = mz[::-1].copy(), None if mz2 is None else mz2[::-1].copy()
    part = torch.cat(parts) if truth else None
    return x, y, z, module.to(torch.int32), offsets, mz, mz2, part


def _alignment(case, seed):
    """Hits displaced by unknown module placements, the particles' hit lists
    (three hits or more, in traversal order) and a current alignment."""
    x, y, z, module, _, mz, _, part = _events(case, seed, truth=True)
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7919)
    M = len(mz)
    place = torch.randn(M, 6, generator=g, device="cuda", dtype=torch.float64)
    place *= torch.tensor([0.01] * 3 + [1.0e-4] * 3, device="cuda", dtype=torch.float64)
    # measured position: the placement applied inversely about the plane centre
    # (first order in the angles, then rounded to the stored fp32)
    m = module.long()
    zc = torch.tensor(mz, device="cuda")[m]
    p = place.float()[m]
    dx, dy, dz = x - p[:, 0], y - p[:, 1], z - zc - p[:, 2]
    a, b, c = p[:, 3], p[:, 4], p[:, 5]
    x, y, z = dx + c * dy - b * dz, dy - c * dx + a * dz, zc + dz + b * dx - a * dy
    order = torch.sort((part << 6) | m)[1]
    order = order[int((part < 0).sum()):]
    n = torch.bincount(part[order])
    order = order[n[part[order]] >= 3]
    n = n[n >= 3]
    ho = torch.zeros(n.numel() + 1, dtype=torch.int32, device="cuda")
    ho[1:] = torch.cumsum(n, 0)
    align = 0.5 * place
    return x, y, z, module, ho, order.to(torch.int32), align, mz


# ------------------------------------------------------------ the calls ---


def _means(case):
    """Mean tracks and hits of a case: a track crosses about 20 planes."""
    tracks = case["events"] * case["pv_mean"] * case["tracks"] * (1.0 + case["backward"])
    return tracks, 20.1 * tracks * (0.5 if case["pairs"] else 1.0)


def _capacity(case):
    """Hits that the program's output buffers hold: sized once for batches of
    this kind, above the spread of the vertices (about 560 hits each)."""
    return int(1.1 * _means(case)[1] + 4000.0 * math.sqrt(case["events"] * case["pv_mean"]))


class _State:
    """What the program keeps; a server is closed before its handle."""

    server = None
    handle = None

    def __del__(self):
        if self.server is not None:
            self.server.close()
        if self.handle is not None:
            self.handle.close()


def prepare(case, seed):
    s = _State()
    s.entry = case["entry"]
    if s.entry in ("align", "align_step"):
        *s.args, s.align, mz = _alignment(case, seed)
        s.handle = sbt.sbt_create(mz, sbt.default_config(hit_sigma=SIGMA))
        if s.entry == "align_step":
            s.align.requires_grad_(True)
        return s
    x, y, z, module, offsets, mz, mz2, _ = _events(case, seed)
    cap = _capacity(case)
    cfg = sbt.default_config(fp16_hits=int(case["fp16"]), gec_max_hits=int(case["cut"]), k_doublets=int(case["k"]))
    s.handle = sbt.sbt_create(mz, cfg, module_z2=mz2)
    s.args = (x, y, z, module, offsets)
    E = offsets.numel() - 1
    if case.get("tuned"):
        sbt.sbt_autotune(s.handle, *s.args)
    if s.entry == "host":
        s.args = tuple(a.cpu().pin_memory() for a in s.args)
        s.out = sbt.TrackOutput.allocate(E, cap, pin_memory=True)
    elif s.entry == "serve":
        o = offsets.cpu().numpy()
        hx, hy, hz, hm = (a.cpu().numpy() for a in s.args[:4])
        s.args = [tuple(a[o[e]:o[e + 1]] for a in (hx, hy, hz, hm)) for e in range(E)]
        s.server = sbt.Server(s.handle, 1 << 30)
        s.out = {"status": np.zeros(E, np.int32), "hit_offsets": np.zeros(E + cap // 3 + 1, np.int32),
                 "track_hits": np.zeros(cap, np.int32), "params": np.zeros((cap // 3, 4), np.float32),
                 "chi2": np.zeros(cap // 3, np.float32), "n_tracks": np.zeros(E, np.int32)}
    else:
        s.out = sbt.TrackOutput.allocate(E, cap)
    return s


def run(state):
    s = state
    if s.entry == "align":
        return sbt.sbt_fit_adjoint(s.handle, *s.args, s.align)
    if s.entry == "align_step":
        s.align.grad = None
        loss = sbt.alignment_chi2(s.handle, *s.args, s.align)
        loss.backward()
        return loss, s.align.grad
    if s.entry == "serve":
        for i, a in enumerate(s.args):
            s.server.submit(i, *a)
        done = []
        while len(done) < len(s.args):
            done += s.server.poll(timeout_s=5.0)
        done.sort(key=lambda r: r.request_id)
        for key, buf in s.out.items():
            if key == "status":
                buf[:] = [r.status for r in done]
            elif key == "n_tracks":
                buf[:] = [len(r.chi2) for r in done]
            else:
                got = np.concatenate([getattr(r, key) for r in done])
                buf[:len(got)] = got
        return s.out
    call = dict(plain=sbt.sbt_reconstruct, batched=sbt.sbt_reconstruct_batched, host=sbt.sbt_reconstruct_host,
                noalloc=sbt.sbt_reconstruct_noalloc)[s.entry]
    return vars(call(s.handle, *s.args, out=s.out))


def work(case):
    """Hits in (16 bytes), hit lists out (4) and 32 bytes a track; the adjoint
    reads hits and lists and does about 80 fp64 operations a hit."""
    tracks, hits = _means(case)
    if case["entry"].startswith("align"):
        return {"bytes": 20.0 * hits + 4.0 * tracks, "flops": 80.0 * hits}
    return {"bytes": 20.0 * hits + 32.0 * tracks, "flops": 0.0}


def tolerance(case):
    # decisions and fits are fixed bit by bit; the adjoint's value and gradient
    # are fp64 sums: residuals of 0.01 mm on coordinates of 40 mm leave up to
    # 4e-14 against 64-bit sums in another order, more on a handful of tracks
    return {"rel": 4.0e-13} if case["entry"].startswith("align") else "exact"


# ---------------------------------------------------------- in 64 bits ---


def exact(case, seed):
    if not case["entry"].startswith("align"):
        return None  # the track sets are decided in fp32: no value in 64 bits
    x, y, z, module, ho, th, align, mz = _alignment(case, seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    a = align.clone().requires_grad_(True)
    ca, sa, cb, sb = torch.cos(a[:, 3]), torch.sin(a[:, 3]), torch.cos(a[:, 4]), torch.sin(a[:, 4])
    cg, sg = torch.cos(a[:, 5]), torch.sin(a[:, 5])
    one, nil = torch.ones_like(ca), torch.zeros_like(ca)

    def mat(*rows):
        return torch.stack([torch.stack(r, -1) for r in rows], -2)

    R = (mat((cg, -sg, nil), (sg, cg, nil), (nil, nil, one)) @ mat((cb, nil, sb), (nil, one, nil), (-sb, nil, cb))
         @ mat((one, nil, nil), (nil, ca, -sa), (nil, sa, ca)))
    zc = torch.tensor(mz, **f64)
    sigma = float(np.float32(SIGMA))  # the library stores it so
    value, grad = torch.zeros(1, **f64), torch.zeros_like(align)
    n_tracks = ho.numel() - 1
    for t0 in range(0, n_tracks, 400000):  # bounded temporaries
        t1 = min(n_tracks, t0 + 400000)
        h = th[int(ho[t0]):int(ho[t1])].long()
        n = (ho[t0 + 1:t1 + 1] - ho[t0:t1]).long()
        seg = torch.repeat_interleave(torch.arange(t1 - t0, device="cuda"), n)
        m = module[h].long()
        v = torch.stack([x[h].double(), y[h].double(), z[h].double() - zc[m]], -1)
        p = (R[m] @ v[:, :, None])[:, :, 0] + a[m, :3]
        p = p + torch.nn.functional.pad(zc[m][:, None], (2, 0))

        def mean(q):
            return torch.zeros(t1 - t0, **f64).index_add(0, seg, q) / n

        dx, dy, dz = (p[:, i] - mean(p[:, i])[seg] for i in range(3))
        szz = mean(dz * dz)
        rx, ry = dx - (mean(dz * dx) / szz)[seg] * dz, dy - (mean(dz * dy) / szz)[seg] * dz
        c = ((rx * rx + ry * ry) / sigma ** 2).sum()
        (part,) = torch.autograd.grad(c, a, retain_graph=True)
        grad += part
        value += c.detach()
    return (value[0], grad) if case["entry"] == "align_step" else (value, grad)
