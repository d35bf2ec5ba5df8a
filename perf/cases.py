"""Performance cases: what programs have the track finder and fitter do.

Every case goes through the public calls of ``Tracker``, ``KFFitChi2`` or
``kf_remove_duplicates_noalloc``.  Events are simulated on the GPU from the
seed alone, with the distributions of the repository's own workloads: tracks
from the origin with pT uniform in 0.5-10 GeV, up to 17 barrel layers (radii
4-110 cm, 0.02 X0 each, Highland scattering), optional endcap disks, Gaussian
hit smearing, uniform noise hits, seeds from the true hits of three layers.
``exact`` restates the method in 64 bits with plain torch.

Fields of a case:
  call       event (plain calls, device arrays), host (the same from and to
             host arrays), batch (replay of a captured graph), fit (re-fit of
             given hit lists), gradient (autograd of the fit's chi2), dedup
             (allocation-free duplicate removal)
  events, tracks, tracks_min   events and generated tracks per event (uniform
             between tracks_min and tracks)
  layers, eta, noise, disks    detector and event shape (disks per side)
  cands      candidates kept per seed
  dup_seeds  second seeds, on layers 2-4, for this share of the tracks
  clean      seed cleaning and kinematic pre-cuts of duplicate removal
  options    material map, parameterized field and energy loss
  adjoint    the graph also takes the gradient of the kept tracks' chi2
  stride     hits between the forward checkpoints of the gradient
"""
import math

import numpy as np
import torch

from paper_1906_11744_gb300 import KF_FIT_GIVEN, Tracker, _lib, kf_get_gradient, make_config, make_detector
from paper_1906_11744_gb300.autograd import KFFitChi2

K_FIELD = 0.00299792458  # 1/rho [1/cm] = K_FIELD * B[T] / pT[GeV]
M_PION = 0.13957


def _f4(v):  # the library takes its settings in 32 bits
    return float(np.float32(v))


BZ, Z_MAX, X0, SIGMA_RPHI, SIGMA_Z, SIGMA_R = (_f4(v) for v in (3.8, 120.0, 0.02, 0.01, 0.1, 0.1))
DISK_RMIN, DISK_RMAX, ETA_BARREL = 15.0, 110.0, _f4(0.9)
PRIOR_VAR = (1.0e-2, 1.0e-2, 1.0e-1, 1.0e-2, 1.0e-4, 4.0e-4)
CHI2_CUT, MAX_HOLES, DUP_FRAC = 30.0, 3, 0.5
FIELD = dict(field_cz=_f4(-0.10 / 120.0 ** 2), field_cr=_f4(-0.05 / 110.0 ** 2))
ELOSS = _f4(7e-4)
CLEAN = dict(seed_clean=1, seed_deta=0.01, seed_dphi=0.01, seed_dpt=0.2, seed_min_shared=0, dup_deta=0.02,
             dup_dphi=0.02, dup_dpt=0.3)
F8 = torch.float64


def _case(call, **kw):
    c = dict(call=call, events=1, tracks=2500, tracks_min=0, layers=17, eta=1.5, noise=0.1, disks=0, cands=6,
             dup_seeds=0.0, clean=False, options=False, adjoint=False, stride=1)
    c.update(kw)
    c["tracks_min"] = c["tracks_min"] or c["tracks"]
    return c


def listed():
    return [
        # one sparse event, as when the finder is tried out or called per region: launches and latency
        dict(_case("event", tracks=100, layers=10, eta=1.0, noise=0.0), name="event_100"),
        # one PU-50 event found, cleaned of duplicates and fitted, event by event
        dict(_case("event", tracks=2500), name="event_pu50"),
        # one PU-200 event from and to host memory, as a trigger or reconstruction job runs it
        dict(_case("host", tracks=8000, noise=0.2, cands=10), name="host_pu200"),
        # one event with the endcap disks searched for the forward half of its seeds
        dict(_case("event", tracks=2500, eta=2.4, disks=7), name="event_endcap"),
        # a few events with the full detector description (odd sizes): material map, varying field, energy loss
        dict(_case("event", events=5, tracks=1777, layers=13, options=True), name="event_options"),
        # doubled seeds: seed cleaning and kinematic duplicate criteria over a small batch
        dict(_case("event", events=8, tracks=8000, noise=0.2, cands=10, dup_seeds=0.1, clean=True), name="event_clean"),
        # a batch of very uneven events through one captured graph
        dict(_case("batch", events=64, tracks=10000, tracks_min=1000), name="batch_mixed"),
        # barrel and endcap batch with the alignment gradient
        dict(_case("batch", events=20, tracks=8000, eta=2.4, noise=0.2, disks=7, cands=10, adjoint=True),
             name="batch_endcap"),
        # the largest batch: 100 PU-200 events with the alignment gradient
        dict(_case("batch", events=100, tracks=8000, noise=0.2, cands=10, adjoint=True), name="batch_pu200"),
        # an alignment job's inner step: chi2 of given tracks and its gradient through autograd
        dict(_case("gradient", tracks=10000, noise=0.0, stride=4), name="gradient_10k"),
        # re-fit of the tracks of many events with given hit lists
        dict(_case("fit", events=30, tracks=6000, noise=0.0), name="fit_180k"),
        # duplicate removal for a host program that allows no device allocation
        dict(_case("dedup", tracks=8000, noise=0.2, dup_seeds=0.1), name="dedup_8k"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(("event", "event", "event", "host", "batch", "batch", "fit", "gradient", "dedup"))
    kw = dict(layers=rng.randint(8, 17), eta=round(rng.uniform(0.8, 1.5), 2), noise=round(rng.uniform(0.0, 0.25), 2),
              cands=rng.choice((4, 5, 6, 6, 8, 10, 10)))
    if call == "event":
        kw.update(events=_spread(rng, 1, 12), tracks=_spread(rng, 80, 8000))
        kind = rng.choice(("plain", "plain", "disks", "options", "clean"))
        if kind == "disks":
            kw.update(disks=rng.randint(2, 7), eta=2.4, layers=17)
        elif kind == "options":
            kw.update(options=True)
        elif kind == "clean":
            kw.update(clean=True, dup_seeds=0.1)
    elif call == "host":
        kw.update(tracks=_spread(rng, 300, 9000))
    elif call == "batch":
        tracks = _spread(rng, 200, 8000)
        kw.update(events=max(1, min(64, _spread(rng, 2000, 300000) // tracks)), tracks=tracks,
                  tracks_min=max(1, int(tracks * rng.choice((0.1, 0.5, 1.0)))), adjoint=rng.random() < 0.5)
        if rng.random() < 0.3:
            kw.update(disks=rng.randint(2, 7), eta=2.4, layers=17)
    elif call == "fit":
        kw.update(events=rng.randint(1, 20), tracks=_spread(rng, 200, 9000))
    elif call == "gradient":
        kw.update(events=rng.randint(1, 4), tracks=_spread(rng, 200, 15000), stride=rng.choice((1, 1, 2, 4)))
    else:
        kw.update(tracks=_spread(rng, 100, 10000), dup_seeds=round(rng.uniform(0.02, 0.3), 2))
    return _case(call, **kw)


# ---------------------------------------------------------------- detector
def _radii(case):
    n, r_max = case["layers"], 100.0 if case["layers"] <= 10 else 110.0
    return [_f4(4.0 + (r_max - 4.0) * i / (n - 1)) for i in range(n)]


def _disk_z(case):
    return [130.0 + 20.0 * k for k in range(case["disks"])]


def _field_terms(case):
    return (FIELD["field_cz"], FIELD["field_cr"]) if case["options"] else (0.0, 0.0)


def _material(case, seed):
    r = np.random.default_rng([seed, 17])
    return r.uniform(0.01, 0.03, size=(case["layers"], 9)).astype(np.float32) if case["options"] else None


def _planes(case):
    """(surface, z) of the disks: the +z side, then the -z side."""
    z = _disk_z(case)
    return [(case["layers"] + i, v) for i, v in enumerate(z + [-v for v in z])]


# ---------------------------------------------------------------- the model in 64 bits
def _to_cylinder(p, b, radius):
    """Helix (p [..., 6] in the field b) to its first crossing of the cylinder, from inside it: (state, crosses)."""
    x, y, z, k, phi, th = p.unbind(-1)
    h = -K_FIELD * b * k
    c, s = torch.cos(phi), torch.sin(phi)
    a_, b_ = (x * c + y * s) * h, (y * c - x * s) * h + 1.0
    e = 0.5 * h * h * (radius * radius - x * x - y * y)
    disc = a_ * a_ + e * (2.0 * b_ - e)
    sg = torch.sign(h)
    psi = 2.0 * torch.atan2(e, a_ * sg + torch.sqrt(disc.clamp(min=1e-14)))
    psi = torch.where(psi <= 0.0, psi + 2.0 * math.pi, psi) * sg
    return _along(p, h, psi), disc > 1e-14


def _to_plane(p, b, zd):
    """Helix to the plane z = zd, forwards and within half a turn: (state, crosses)."""
    h = -K_FIELD * b * p[..., 3]
    arc = (zd - p[..., 2]) * torch.tan(p[..., 5])
    q = _along(p, h, h * arc)
    return q, (arc > 0) & (torch.abs(h * arc) < math.pi)


def _along(p, h, psi):
    x, y, z, k, phi, th = p.unbind(-1)
    c, s = torch.cos(phi), torch.sin(phi)
    sx, cx = torch.sin(psi) / h, 2.0 * torch.sin(0.5 * psi) ** 2 / h
    return torch.stack([x + c * sx - s * cx, y + s * sx + c * cx, z + psi / h / torch.tan(th), k, phi + psi, th], -1)


def _lost(p, e, disk):
    """q/pT after the mean energy loss e of a surface."""
    x, y, z, k, phi, th = p.unbind(-1)
    st = torch.sin(th)
    mom = 1.0 / (torch.abs(k) * st)
    en = torch.sqrt(mom * mom + M_PION ** 2)
    slope = torch.abs(torch.cos(th)) if disk else st * torch.abs(torch.cos(phi - torch.atan2(y, x)))
    de = torch.minimum(e * en * en / (mom * mom * slope), 0.5 * (en - M_PION))
    k2 = k * mom / torch.sqrt((en - de) ** 2 - M_PION ** 2)
    return torch.stack([x, y, z, k2, phi, th], -1)


def _highland(k, th, thickness):
    mom = 1.0 / (torch.abs(k) * torch.sin(th))
    beta = mom / torch.sqrt(mom * mom + M_PION ** 2)
    return 0.0136 / (beta * mom) * torch.sqrt(thickness) * (1.0 + 0.038 * torch.log(thickness))


class _Model:
    """Steps of the Kalman filter over states p [n, 6] and covariances C [n, 6, 6]."""

    def __init__(self, case, seed, dev):
        self.radii, self.case = _radii(case), case
        self.planes = dict(_planes(case))
        self.n_surf = case["layers"] + 2 * case["disks"]
        self.cz, self.cr = _field_terms(case)
        m = _material(case, seed)
        self.x0 = None if m is None else torch.from_numpy(m).to(dev, F8)
        self.eloss = ELOSS if case["options"] else 0.0

    def field(self, p):
        return BZ * (1.0 + self.cz * p[..., 2] ** 2 + self.cr * (p[..., 0] ** 2 + p[..., 1] ** 2))

    def propagate(self, p, C, s):
        """To surface s: (p, C, crosses within the surface)."""
        def step(q, b):
            return _to_plane(q, b, self.planes[s])[0] if s in self.planes else _to_cylinder(q, b, self.radii[s])[0]

        b = self.field(p)
        if s in self.planes:
            q, ok = _to_plane(p, b, self.planes[s])
        else:
            q, ok = _to_cylinder(p, b, self.radii[s])
        J = torch.func.vmap(torch.func.jacfwd(step))(p, b)
        return q, J @ C @ J.transpose(-1, -2), ok

    def within(self, q, s):
        if s in self.planes:
            r = torch.hypot(q[..., 0], q[..., 1])
            return (r >= DISK_RMIN) & (r <= DISK_RMAX)
        return torch.abs(q[..., 2]) <= Z_MAX

    def frame(self, p, C, s):
        """(H [n, 2, 6], S^-1 [n, 2, 2]) of the measurement at the prediction."""
        r = torch.hypot(p[..., 0], p[..., 1])
        c, sn, o = p[..., 0] / r, p[..., 1] / r, torch.zeros_like(r)
        second = [c, sn, o, o, o, o] if s in self.planes else [o, o, o + 1.0, o, o, o]
        H = torch.stack([torch.stack([-sn, c, o, o, o, o], -1), torch.stack(second, -1)], -2)
        v = torch.tensor([SIGMA_RPHI ** 2, (SIGMA_R if s in self.planes else SIGMA_Z) ** 2], dtype=F8, device=p.device)
        S = H @ C @ H.transpose(-1, -2) + torch.diag(v)
        det = S[..., 0, 0] * S[..., 1, 1] - S[..., 0, 1] ** 2
        inv = torch.stack([torch.stack([S[..., 1, 1], -S[..., 0, 1]], -1), torch.stack([-S[..., 0, 1], S[..., 0, 0]], -1)], -2)
        return H, inv / det[..., None, None]

    def update(self, p, C, m, s):
        """With the hits m [n, 3]: (p, C, chi2)."""
        H, Si = self.frame(p, C, s)
        r = (H @ (torch.nn.functional.pad(m, (0, 3)) - p)[..., None])
        G = C @ H.transpose(-1, -2) @ Si
        return p + (G @ r)[..., 0], C - G @ (H @ C), (r.transpose(-1, -2) @ Si @ r)[..., 0, 0]

    def scatter(self, p, C, s):
        disk = s in self.planes
        if disk:
            x0, slope = X0, torch.abs(torch.cos(p[..., 5]))
        else:
            slope = torch.sin(p[..., 5]) * torch.abs(torch.cos(p[..., 4] - torch.atan2(p[..., 1], p[..., 0])))
            x0 = X0
            if self.x0 is not None:
                m = self.x0[s]
                u = ((p[..., 2] + Z_MAX) * (len(m) - 1) / (2 * Z_MAX)).clamp(0, len(m) - 1)
                i = u.detach().floor().long().clamp(max=len(m) - 2)
                x0 = m[i] + (u - i) * (m[i + 1] - m[i])
        v = _highland(p[..., 3], p[..., 5], x0 / slope) ** 2
        o = torch.zeros_like(v)
        C = C + torch.diag_embed(torch.stack([o, o, o, o, v / torch.sin(p[..., 5]) ** 2, v], -1))
        if self.eloss > 0 and not disk:
            F = torch.func.vmap(torch.func.jacfwd(lambda q: _lost(q, self.eloss, disk)))(p)
            p, C = _lost(p, self.eloss, disk), F @ C @ F.transpose(-1, -2)
        return p, C


def _pick(mask, a, b):
    return torch.where(mask.reshape(mask.shape + (1,) * (a.dim() - mask.dim())), a, b)


def _aligned(model, m, s, align):
    """Hits m [..., 3] of barrel layer s corrected for its alignment offsets."""
    if s in model.planes:
        return m
    a = -align[s, 0] / model.radii[s]
    c, sn = torch.cos(a), torch.sin(a)
    return torch.stack([c * m[..., 0] - sn * m[..., 1], sn * m[..., 0] + c * m[..., 1], m[..., 2] - align[s, 1]], -1)


def _fit64(model, p, C, rows, hits, align):
    """Kalman fit over rows [n, n_surf] of hit indices (-1: none): (p, C, chi2, fitted)."""
    chi2 = torch.zeros(len(p), dtype=F8, device=p.device)
    ok = torch.ones(len(p), dtype=torch.bool, device=p.device)
    started = torch.zeros_like(ok)
    left = (rows >= 0).sum(1)
    for s in range(model.n_surf):
        has = (rows[:, s] >= 0) & ok
        if not bool(has.any()):
            continue
        q, D, cross = model.propagate(p, C, s)
        ok = ok & ~(has & started & ~cross)
        has = has & ok
        move = has & started
        q, D = _pick(move, q, p), _pick(move, D, C)
        m = _pick(has, _aligned(model, hits[rows[:, s].clamp(min=0)], s, align), q[:, :3].detach())
        u, U, c2 = model.update(q, D, m, s)
        left = left - has.long()
        w, W = model.scatter(u, U, s)
        u, U = _pick(left > 0, w, u), _pick(left > 0, W, U)
        p, C, chi2 = _pick(has, u, p), _pick(has, U, C), chi2 + torch.where(has, c2, torch.zeros_like(c2))
        started = started | has
    return p, C, chi2, ok


def _find64(model, ev, N, align):
    """Combinatorial finding of one event, every hit of a surface tested: (rows [n, n_surf], n, chi2, p, C)."""
    hits, lay, dev = ev["hits"], ev["layer"].long(), ev["hits"].device
    at = [torch.nonzero(lay == s)[:, 0] for s in range(model.n_surf)]
    cor = [_aligned(model, hits[i], s, align) for s, i in enumerate(at)]
    outs = []
    for lo in range(0, len(ev["p"]), 1024):
        p, C, sh = ev["p"][lo:lo + 1024], ev["C"][lo:lo + 1024], ev["seed_hits"][lo:lo + 1024].long()
        n = len(p)
        srow = torch.full((n, model.n_surf), -1, dtype=torch.long, device=dev)
        srow.scatter_(1, lay[sh], sh)
        last = lay[sh[:, 2]]
        eta = -torch.log(torch.tan(0.5 * p[:, 5]))
        p, C, chi2, ok = _fit64(model, p, C, srow, hits, align)
        for s in range(model.case["layers"]):  # the scattering of the third seed hit's layer
            w, W = model.scatter(p, C, s)
            p, C = _pick((last == s) & ok, w, p), _pick((last == s) & ok, W, C)
        fwd = (torch.abs(eta) >= ETA_BARREL) & (model.case["disks"] > 0)
        S = dict(p=p[:, None].repeat(1, N, 1), C=C[:, None].repeat(1, N, 1, 1), chi2=chi2[:, None].repeat(1, N),
                 nf=torch.full((n, N), 3, device=dev), holes=torch.zeros((n, N), dtype=torch.long, device=dev),
                 done=~ok[:, None].repeat(1, N), rows=srow[:, None].repeat(1, N, 1))
        occ = torch.zeros((n, N), dtype=torch.bool, device=dev)
        occ[:, 0] = True
        for s in range(model.n_surf):
            z = model.planes.get(s)
            mine = (s > last) if z is None else (fwd & ((eta < 0) == (z < 0)))
            q, D, cross = model.propagate(S["p"].reshape(-1, 6), S["C"].reshape(-1, 6, 6), s)
            cross = (cross & model.within(q, s)).reshape(n, N)
            live = occ & ~S["done"] & mine[:, None]
            step = live & cross
            S["done"] = S["done"] | (live & ~cross & ~fwd[:, None])
            H, Si = model.frame(q, D, s)
            m = cor[s]
            r = (torch.nn.functional.pad(m, (0, 3)) @ H.transpose(-1, -2)) - (H @ q[..., None])[..., 0][:, None]
            c2 = Si[:, None, 0, 0] * r[..., 0] ** 2 + 2 * Si[:, None, 0, 1] * r[..., 0] * r[..., 1] + \
                Si[:, None, 1, 1] * r[..., 1] ** 2
            del r
            near = (m[:, :2] @ q[:, :2].T).T > 0
            c2 = torch.where((c2 < CHI2_CUT) & near & step.reshape(-1, 1), c2, math.inf)
            k = min(N, c2.shape[1])
            best, which = torch.topk(c2, k, dim=1, largest=False) if k else (c2[:, :0], c2[:, :0].long())
            del c2, near
            best, which = best.reshape(n, N, k), at[s][which].reshape(n, N, k)
            good = torch.isfinite(best)
            tail = occ & (~step | (S["holes"] < MAX_HOLES) | ~good.any(-1))
            stop = step & (S["holes"] >= MAX_HOLES) & ~good.any(-1)
            slot = torch.arange(N, device=dev)[None, :, None].expand(n, N, k + 1).reshape(n, -1)
            valid = torch.cat([good, tail[..., None]], -1).reshape(n, -1)
            nf = torch.cat([S["nf"][..., None] + good.long(), S["nf"][..., None]], -1).reshape(n, -1)
            ch = torch.cat([S["chi2"][..., None] + best, S["chi2"][..., None]], -1).reshape(n, -1)
            hit = torch.cat([which, torch.full_like(slot.reshape(n, N, k + 1)[..., :1], -1)], -1).reshape(n, -1)
            order = torch.argsort((slot * 2 + (hit < 0)) * (len(hits) + 1) + hit, dim=1, stable=True)
            for key in (ch, -nf, (~valid).long()):  # least significant first
                order = order.gather(1, torch.argsort(key.gather(1, order), dim=1, stable=True))
            order = order[:, :N]
            par, hit, valid = slot.gather(1, order), hit.gather(1, order), valid.gather(1, order)
            q, D = _pick(step & ~stop, q.reshape(n, N, 6), S["p"]), _pick(step & ~stop, D.reshape(n, N, 6, 6), S["C"])
            row = torch.arange(n, device=dev)[:, None]
            hole = valid & (hit < 0) & (step & ~stop)[row, par]
            T = {key: v[row, par] for key, v in S.items()}
            T["done"] = T["done"] | stop[row, par]
            q, D = q[row, par].reshape(-1, 6), D[row, par].reshape(-1, 6, 6)
            got = valid & (hit >= 0)
            u, U, _ = model.update(q, D, _aligned(model, hits[hit.clamp(min=0).reshape(-1)], s, align), s)
            q, D = _pick(got.reshape(-1), u, q), _pick(got.reshape(-1), U, D)
            w, W = model.scatter(q, D, s)
            do = (got | hole).reshape(-1)
            T["p"], T["C"] = _pick(do, w, q).reshape(n, N, 6), _pick(do, W, D).reshape(n, N, 6, 6)
            T["chi2"], T["nf"] = ch.gather(1, order), nf.gather(1, order)
            T["holes"] = T["holes"] + hole.long()
            T["rows"][..., s] = torch.where(got, hit, T["rows"][..., s])
            keep = mine[:, None].expand(n, N)
            S = {key: _pick(keep, T[key], S[key]) for key in S}
            occ = _pick(keep, valid, occ)
        outs.append(tuple(S[key][:, 0] for key in ("rows", "nf", "chi2", "p", "C")))
    return tuple(torch.cat(v) for v in zip(*outs))


def _kept64(rows, nf, chi2):
    """Duplicate removal on shared hits, in order of more hits and lower chi2."""
    R, n, c = rows.cpu().numpy(), nf.cpu().numpy(), chi2.cpu().numpy()
    keep, owners = np.zeros(len(R), bool), {}
    for t in sorted(range(len(R)), key=lambda i: (-n[i], c[i], i)):
        mine, shared = R[t][R[t] >= 0].tolist(), {}
        for h in mine:
            for o in owners.get(h, ()):
                shared[o] = shared.get(o, 0) + 1
        if all(v <= DUP_FRAC * min(n[t], n[o]) for o, v in shared.items()):
            keep[t] = True
            for h in mine:
                owners.setdefault(h, []).append(t)
    return torch.from_numpy(keep).to(rows.device)


def _gradient64(model, p, C, rows, hits, align):
    """(chi2, gradients with respect to alignment, hits and seed parameters) of the summed fit chi2."""
    leaves = [v.clone().requires_grad_(True) for v in (align, hits, p)]
    total, grads = 0.0, [torch.zeros_like(v) for v in leaves]
    for lo in range(0, len(p), 8192):
        sl = slice(lo, lo + 8192)
        _, _, chi2, ok = _fit64(model, leaves[2][sl], C[sl], rows[sl], leaves[1], leaves[0])
        part = torch.where(ok, chi2, torch.zeros_like(chi2)).sum()
        for g, d in zip(grads, torch.autograd.grad(part, leaves)):
            g += d
        total = total + part.detach()
    return total, grads


# ---------------------------------------------------------------- events
def _tracks(case):
    """Generated tracks of each event, the same for every seed."""
    r = np.random.default_rng([case["events"], case["tracks"]])
    return r.integers(case["tracks_min"], case["tracks"] + 1, size=case["events"])


def _event_hits(case):
    """Hits of each event, the same for every seed: noise hits make up what its tracks leave."""
    n = _tracks(case)
    return np.ceil(n * _hits_per_track(case) * (1 + case["noise"]) + 12 * np.sqrt(n))


def _simulate(case, seed):
    """Events of a case on the GPU: hits, layers, seeds, offsets and the true rows [tracks, n_surf] (event-local)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed) * 1000003 + 17)
    uni = lambda n, a, b: torch.rand(n, generator=gen, device=dev, dtype=F8) * (b - a) + a  # noqa: E731
    nrm = lambda n: torch.randn(n, generator=gen, device=dev, dtype=F8)  # noqa: E731
    E, radii, cz, cr = case["events"], _radii(case), *_field_terms(case)
    per = _tracks(case)
    ev = torch.repeat_interleave(torch.arange(E, device=dev), torch.from_numpy(per).to(dev))
    n = len(ev)
    eta, q = uni(n, -case["eta"], case["eta"]), torch.sign(uni(n, -1, 1) + 1e-300)
    p = torch.stack([0.01 * nrm(n), 0.01 * nrm(n), 0.01 * nrm(n), q / uni(n, 0.5, 10.0), uni(n, -math.pi, math.pi),
                     2 * torch.atan(torch.exp(-eta))], -1)
    fits = case["call"] in ("fit", "gradient")
    align = torch.randn(len(radii), 2, generator=gen, device=dev, dtype=F8) * (0.005 if fits else 0.0)
    align = align.float().double()
    field = lambda v: BZ * (1 + cz * v[:, 2] ** 2 + cr * (v[:, 0] ** 2 + v[:, 1] ** 2))  # noqa: E731
    alive = torch.ones(n, dtype=torch.bool, device=dev)
    surfaces = [(s, None) for s in range(len(radii))] + _planes(case)
    hx, hev, hlay, htrk = [], [], [], []
    for s, zd in surfaces:
        if zd is None:
            w, r0, ok = p, torch.hypot(p[:, 0], p[:, 1]), alive
            for k in range(1, 9 if case["options"] else 2):  # a varying field is followed in eight steps
                w, c = _to_cylinder(w, field(w), r0 + (radii[s] - r0) * k / 8 if case["options"] else radii[s])
                ok = ok & c
            ok = ok & (torch.abs(w[:, 2]) <= Z_MAX)
            alive = ok
            ang = torch.atan2(w[:, 1], w[:, 0])
            a = ang + (SIGMA_RPHI * nrm(n) + align[s, 0]) / radii[s]
            m = torch.stack([radii[s] * torch.cos(a), radii[s] * torch.sin(a), w[:, 2] + SIGMA_Z * nrm(n) + align[s, 1]], -1)
            path = X0 / torch.abs(torch.sin(w[:, 5]) * torch.cos(w[:, 4] - ang))
        else:
            w, ok = _to_plane(p, field(p), zd)
            r, ang = torch.hypot(w[:, 0], w[:, 1]), torch.atan2(w[:, 1], w[:, 0])
            ok = ok & (r >= DISK_RMIN) & (r <= DISK_RMAX)
            a, rr = ang + SIGMA_RPHI * nrm(n) / r, r + SIGMA_R * nrm(n)
            m = torch.stack([rr * torch.cos(a), rr * torch.sin(a), torch.full_like(r, zd)], -1)
            path = X0 / torch.abs(torch.cos(w[:, 5]))
        th0 = torch.nan_to_num(_highland(w[:, 3], w[:, 5], path))
        kick = torch.zeros_like(w)
        kick[:, 4], kick[:, 5] = nrm(n) * th0 / torch.sin(w[:, 5]), nrm(n) * th0
        p = _pick(ok, w + kick, p)
        idx = torch.nonzero(ok)[:, 0]
        hx.append(m[idx])
        hev.append(ev[idx])
        htrk.append(idx)
        hlay.append(torch.full((len(idx),), s, dtype=torch.int32, device=dev))
    # noise hits, as the true ones spread over the surfaces, fill each event up to its number of hits
    true = torch.stack([torch.bincount(v, minlength=E) for v in hev], 1).double()
    noisy = (torch.from_numpy(_event_hits(case)).to(dev) - true.sum(1)).clamp(min=0)
    upto = torch.floor(noisy[:, None] * true.cumsum(1) / true.sum(1, keepdim=True) + 1e-6).long()
    share = torch.diff(upto, dim=1, prepend=torch.zeros_like(upto[:, :1])).reshape(-1)
    cell = torch.repeat_interleave(torch.arange(len(share), device=dev), share)
    nev, ns = cell // len(surfaces), cell % len(surfaces)
    disk = torch.tensor([zd is not None for _, zd in surfaces], device=dev)[ns]
    at = torch.tensor([radii[s] if zd is None else zd for s, zd in surfaces], dtype=F8, device=dev)[ns]
    f, v = uni(len(nev), -math.pi, math.pi), uni(len(nev), 0, 1)
    r = torch.where(disk, torch.sqrt(DISK_RMIN ** 2 + v * (DISK_RMAX ** 2 - DISK_RMIN ** 2)), at)
    zz = torch.where(disk, at, (2 * v - 1) * Z_MAX)
    hx.append(torch.stack([r * torch.cos(f), r * torch.sin(f), zz], -1))
    hev.append(nev)
    htrk.append(torch.full_like(nev, -1))
    hlay.append(ns.int())
    hits, hev, htrk, lay = torch.cat(hx).float(), torch.cat(hev), torch.cat(htrk), torch.cat(hlay)
    perm = torch.randperm(len(hev), generator=gen, device=dev)  # the order of an event's hits says nothing
    perm = perm[torch.argsort(hev[perm], stable=True)]
    hits, hev, htrk, lay = hits[perm], hev[perm], htrk[perm], lay[perm]
    hit_off = torch.cat([torch.zeros(1, dtype=torch.long, device=dev), torch.bincount(hev, minlength=E).cumsum(0)])
    rows = torch.full((n, len(surfaces)), -1, dtype=torch.long, device=dev)
    true = torch.nonzero(htrk >= 0)[:, 0]
    rows[htrk[true], lay[true].long()] = true - hit_off[hev[true]]
    trk = torch.nonzero((rows[:, :3] >= 0).all(1))[:, 0]
    sh, srow, sev = rows[trk, :3], trk, ev[trk]
    if case["dup_seeds"] and case["layers"] > 3:
        mix = torch.randperm(n, generator=gen, device=dev)
        mix = mix[torch.argsort(ev[mix], stable=True)]
        first = torch.from_numpy(np.cumsum(per) - per).to(dev)
        picked = torch.arange(n, device=dev) - first[ev] < torch.from_numpy(np.round(case["dup_seeds"] * per)).to(dev)[ev]
        extra = torch.sort(mix[picked])[0]
        sh, srow, sev = torch.cat([sh, rows[extra, 1:4]]), torch.cat([srow, extra]), torch.cat([sev, ev[extra]])
        o = torch.argsort(sev, stable=True)
        sh, srow, sev = sh[o], srow[o], sev[o]
    seed_off = torch.cat([torch.zeros(1, dtype=torch.long, device=dev), torch.bincount(sev, minlength=E).cumsum(0)])
    P = hits.double()[sh + hit_off[sev][:, None]]
    (ax, ay, az), (bx, by, _), (cx, cy, c_z) = (P[:, i].unbind(-1) for i in range(3))
    d = 2 * (ax * (by - cy) + bx * (cy - ay) + cx * (ay - by))  # circle through the three hits
    a2, b2, c2 = ax * ax + ay * ay, bx * bx + by * by, cx * cx + cy * cy
    ux, uy = (a2 * (by - cy) + b2 * (cy - ay) + c2 * (ay - by)) / d, (a2 * (cx - bx) + b2 * (ax - cx) + c2 * (bx - ax)) / d
    sg = torch.where((bx - ax) * (cy - by) - (by - ay) * (cx - bx) >= 0, 1.0, -1.0)
    rho = torch.hypot(ax - ux, ay - uy)
    arc = rho * torch.remainder(sg * torch.atan2((ax - ux) * (cy - uy) - (ay - uy) * (cx - ux),
                                                 (ax - ux) * (cx - ux) + (ay - uy) * (cy - uy)), 2 * math.pi)
    params = torch.stack([ax, ay, az, -sg / rho / (K_FIELD * BZ), torch.atan2(sg * (ax - ux), -sg * (ay - uy)),
                          torch.atan2(torch.ones_like(arc), (c_z - az) / arc)]).float().contiguous()
    diag = [i * 6 - i * (i - 1) // 2 for i in range(6)]
    cov = torch.zeros(21, len(sh), device=dev)
    cov[diag] = torch.tensor(PRIOR_VAR, device=dev)[:, None]
    x, y, z = (hits[:, i].contiguous() for i in range(3))
    return dict(x=x, y=y, z=z, layer=lay, params=params, cov=cov, seed_hits=sh.T.int().contiguous(),
                hit_off=hit_off.cpu().numpy().astype(np.int32), seed_off=seed_off.cpu().numpy().astype(np.int32),
                align=align.float(), rows=rows[srow], gen=gen)


def _lists(rows):
    """Hit lists [n, n_surf], -1 padded at the end, and their lengths."""
    order = torch.argsort((rows < 0).int(), dim=1, stable=True)
    return rows.gather(1, order).int().contiguous(), (rows >= 0).sum(1).int()


def _found(case, d):
    """A tracker's found tracks, as a caller of the allocation-free entry point holds them: the true hit lists, some
    of them with a copy that lost or exchanged a few hits."""
    rows, gen = d["rows"].clone(), d["gen"]
    n, dev = len(rows), rows.device
    first = d["params"][0]  # second seeds are copies; they lose hits at random
    lose = torch.rand(rows.shape, generator=gen, device=dev) < 0.08
    rows[lose & (torch.arange(rows.shape[1], device=dev) >= 3)] = -1
    swap = (torch.rand(rows.shape, generator=gen, device=dev) < 0.05) & (rows >= 0)
    other = rows[torch.randperm(n, generator=gen, device=dev)]
    rows = torch.where(swap & (other >= 0), other, rows)
    lists, n_found = _lists(rows)
    chi2 = (torch.randn(n, 2 * rows.shape[1], generator=gen, device=dev) ** 2).sum(1) + first.abs() * 1e-3
    return lists, n_found, chi2


# ---------------------------------------------------------------- the cases
def prepare(case, seed):
    d = _simulate(case, seed)
    s = dict(case=case, d=d)
    if case["call"] == "dedup":
        s["lists"], s["n_found"], s["chi2"] = _found(case, d)
        return s
    opts = dict(eloss=[ELOSS] * case["layers"], **FIELD) if case["options"] else {}
    det = make_detector(_radii(case), [X0] * case["layers"], Z_MAX, BZ, SIGMA_RPHI, SIGMA_Z, disk_z=_disk_z(case),
                        disk_rmin=DISK_RMIN, disk_rmax=DISK_RMAX, disk_x0=X0, sigma_r=SIGMA_R, eta_barrel=ETA_BARREL,
                        **opts)
    cfg = make_config(max_cands=case["cands"], max_holes=MAX_HOLES, chi2_cut=CHI2_CUT, dup_shared_frac=DUP_FRAC,
                      ckpt_stride=case["stride"], **(CLEAN if case["clean"] else {}))
    s["t"] = t = Tracker(det, cfg)
    if case["options"]:
        t.set_material(_material(case, seed))
    t.set_alignment(d["align"])
    if case["call"] == "host":
        for k in ("x", "y", "z", "layer", "params", "cov", "seed_hits"):
            d[k] = d[k].cpu().pin_memory()
    s["stream"] = torch.cuda.Stream() if case["call"] == "batch" else None
    if s["stream"] is not None:
        s["stream"].wait_stream(torch.cuda.current_stream())
    _load(s)
    if case["call"] == "batch":  # a long-running job tunes the launch shape once and keeps the captured graph
        t.autotune(s["stream"])
        t.capture_graph(with_adjoint=case["adjoint"], stream=s["stream"])
    if case["call"] in ("fit", "gradient"):
        s["lists"], s["n_hits"] = _lists(d["rows"])
    if case["call"] == "gradient":
        t.hit_offsets, t.seed_offsets = d["hit_off"], d["seed_off"]
        t.layer_dev, t.cov_dev, t.seed_hits_dev = d["layer"], d["cov"], d["seed_hits"]
        s["leaves"] = [v.clone().requires_grad_(True) for v in
                       (d["align"], torch.stack([d["x"], d["y"], d["z"]], 1), d["params"])]
    return s


def _load(s):
    d, t = s["d"], s["t"]
    t.load_hits(d["hit_off"], d["x"], d["y"], d["z"], d["layer"], s["stream"])
    t.load_seeds(d["seed_off"], d["params"], d["cov"], d["seed_hits"], s["stream"])


def run(s):
    case, d, t = s["case"], s["d"], s.get("t")
    call = case["call"]
    if call == "dedup":
        n, L = s["lists"].shape
        keep = torch.empty(n, dtype=torch.uint8, device="cuda")
        status = torch.empty(1, dtype=torch.int32, device="cuda")
        rc = _lib.kf_remove_duplicates_noalloc(n, L, int(d["hit_off"][-1]), s["lists"], s["n_found"], s["chi2"],
                                               DUP_FRAC, keep, status)
        return dict(rc=rc, keep=keep, status=status)
    if call == "gradient":
        align, hits, seeds = s["leaves"]
        chi2 = KFFitChi2.apply(t, align, hits, seeds, s["lists"], s["n_hits"])
        g = torch.autograd.grad(chi2, s["leaves"])
        return dict(chi2=chi2.detach(), g_align=g[0], g_hits=g[1], g_seed=g[2])
    if call == "fit":
        _load(s)
        t.fit_tracks(KF_FIT_GIVEN, s["lists"], s["n_hits"])
        return t.get_fit("cuda")
    if call == "batch":
        st = s["stream"]
        with torch.cuda.stream(st):
            _load(s)
            t.launch_graph(st)
            out = dict(tracks=t.get_tracks("cuda", st), fit=t.get_fit("cuda", st))
            if case["adjoint"]:
                out["g"] = dict(align=torch.empty(case["layers"], 2, device="cuda"),
                                hits=torch.empty(int(d["hit_off"][-1]), 3, device="cuda"),
                                seed=torch.empty_like(d["params"]))
                kf_get_gradient(t.ctx, out["g"]["align"], out["g"]["hits"], out["g"]["seed"], st)
        return out
    _load(s)
    t.find_tracks()
    t.remove_duplicates()
    t.fit_tracks()
    dev = None if call == "host" else "cuda"
    return dict(tracks=t.get_tracks(dev), fit=t.get_fit(dev))


def _hits_per_track(case):
    """Mean surfaces crossed by a track of the case's pT and |eta| range."""
    eta = np.linspace(0.0, case["eta"], 201)[1:, None]
    pt = np.linspace(0.5, 10.0, 100)[None]
    rho = pt / (K_FIELD * BZ)
    n = 0.0
    for r in _radii(case):
        arc = 2 * rho * np.arcsin(np.minimum(r / (2 * rho), 1.0))
        n += np.mean((r < 2 * rho) & (arc * np.sinh(eta) <= Z_MAX))
    for z in _disk_z(case):
        r = 2 * rho * np.abs(np.sin(np.minimum(z / np.sinh(eta) / (2 * rho), math.pi / 2)))
        n += np.mean((r >= DISK_RMIN) & (r <= DISK_RMAX))
    return float(n)


def work(case):
    tracks, hits, per = float(_tracks(case).sum()), float(_event_hits(case).sum()), _hits_per_track(case)
    seeds, surf = tracks * (1 + case["dup_seeds"]), case["layers"] + 2 * case["disks"]
    fit = 500.0 * seeds * per  # propagation, transport and update per hit
    if case["call"] == "dedup":
        return dict(bytes=seeds * (4 * surf + 9.0), flops=seeds * per)
    state = 4.0 * 28 * seeds + 4.0 * seeds  # parameters, covariance, chi2 and status
    load = 16.0 * hits + 4.0 * 30 * seeds
    grad = 12.0 * hits + 24.0 * seeds
    if case["call"] == "fit":
        return dict(bytes=load + 4.0 * seeds * surf + state, flops=fit)
    if case["call"] == "gradient":
        return dict(bytes=load + 4.0 * seeds * surf + grad, flops=4 * fit)
    # about 620 operations per candidate and surface, four fifths of the candidates' places taken
    find = 620.0 * seeds * 0.8 * case["cands"] * max(per - 3, 1)
    return dict(bytes=load + 4.0 * seeds * surf + 2 * state + (grad if case["adjoint"] else 0),
                flops=find + fit * (4 if case["adjoint"] else 1))


def _upper(C):
    return torch.stack([C[:, i, j] for i in range(6) for j in range(i, 6)])


def exact(case, seed):
    call, n_max = case["call"], case["tracks"]
    fitted = case["events"] * n_max * case["layers"]
    if call == "dedup" or case["clean"]:  # whole numbers; tracks that depend on which of two seeds was kept
        return None
    if call in ("fit", "gradient"):
        if fitted > (4e6 if call == "fit" else 6e5):
            return None
    elif case["events"] * float(n_max) ** 2 * case["cands"] * (case["layers"] + case["disks"]) > 1.2e10 or fitted > 6e5:
        return None  # over about 20 seconds
    d = _simulate(case, seed)
    model, dev = _Model(case, seed, "cuda"), torch.device("cuda")
    align = d["align"].double()
    hits = torch.stack([d["x"], d["y"], d["z"]], 1).double()
    p, C = d["params"].double().T.contiguous(), torch.zeros(d["params"].shape[1], 6, 6, dtype=F8, device=dev)
    C[:, list(range(6)), list(range(6))] = torch.tensor(PRIOR_VAR, device=dev).double()
    so, ho = d["seed_off"], d["hit_off"]
    base = torch.repeat_interleave(torch.from_numpy(ho[:-1].astype(np.int64)), torch.from_numpy(np.diff(so)).long()).to(dev)
    if call in ("fit", "gradient"):
        rows = torch.where(d["rows"] >= 0, d["rows"] + base[:, None], -1)
        if call == "gradient":
            chi2, g = _gradient64(model, p, C, rows, hits, align)
            return dict(chi2=chi2, g_align=g[0], g_hits=g[1], g_seed=g[2].T.contiguous())
        with torch.no_grad():
            q, D, chi2, _ = _fit64(model, p, C, rows, hits, align)
        return dict(params=q.T, cov=_upper(D), chi2=chi2, status=None)
    with torch.no_grad():
        parts, keep = [], []
        for e in range(case["events"]):
            a, b = so[e], so[e + 1]
            ev = dict(hits=hits[ho[e]:ho[e + 1]], layer=d["layer"][ho[e]:ho[e + 1]], p=p[a:b], C=C[a:b],
                      seed_hits=d["seed_hits"][:, a:b].T)
            parts.append(_find64(model, ev, case["cands"], align))
            keep.append(_kept64(*parts[-1][:3]))
        rows, nf, chi2, q, D = (torch.cat(v) for v in zip(*parts))
        keep = torch.cat(keep)
        rows = torch.where(rows >= 0, rows + base[:, None], -1)
        out = dict(tracks=dict(hits=None, n_found=None, chi2=chi2, params=q.T, cov=_upper(D), keep=None))
        fq, fD, fc, _ = _fit64(model, p, C, rows, hits, align)
        zero = keep.double()
        out["fit"] = dict(params=fq.T * zero, cov=_upper(fD) * zero, chi2=fc * zero, status=None)
    if case["adjoint"]:
        _, g = _gradient64(model, p, C, torch.where(keep[:, None], rows, -1), hits, align)
        out["g"] = dict(align=g[0], hits=g[1], seed=g[2].T.contiguous())
    return out
