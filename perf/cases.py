"""Timed workloads of the transport library, each through a public entry point.

``listed()`` names the workloads, ``prepare`` makes what a user's program has
in hand before a call (primaries, a context or server, device buffers),
``run`` is one call with all of its tallies, ``work`` what a call cannot do
without, and ``exact`` the normalised tallies of the thin-column workloads as
plain numpy gives them in 64 bits.

Families:

* ``thin``: beta electrons in a uniform thin column (a few collisions each),
  optionally with a scattering-angle table; one pass, host buffers.
* ``source``: the two-pass source run, one beta electron and one thermal T2+
  per decay in a parabolic column; host buffers or device buffers.
* ``cycles``: the same source with its fields updated in cycles.
* ``chemistry``: the source with T+ chemistry and charge exchange.
* ``thermal``: electrons thermalising on a moving target.
* ``batch``: many source configurations of uneven size through one server.
* ``orbit_ions`` / ``orbit_tube``: full-orbit transport of ions, or of beta
  electrons and ions with their products, in a beam tube.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_10263_gb300 import inputs, karl

FP64, FP32 = karl.FP64, karl.FP32


def listed():
    return [
        # a first look at a thin column: the smallest call, all latency
        {"name": "thin_1e3_fp64", "kind": "thin", "n": 1000, "nz": 1000, "precision": FP64,
         "angular": False},
        # thin column with tabulated elastic angles in the precision form
        {"name": "thin_angular_2e4_fp32", "kind": "thin", "n": 20011, "nz": 1000,
         "precision": FP32, "angular": True},
        # a quick source run while setting parameters: few decays, both passes
        {"name": "source_1e3_fp64", "kind": "source", "n": 1000, "nz": 1000, "column": 5e21,
         "length": 10.0, "precision": FP64, "device": False},
        # an ordinary source run with host buffers
        {"name": "source_1e5_fp64", "kind": "source", "n": 100_000, "nz": 1000, "column": 5e21,
         "length": 10.0, "precision": FP64, "device": False},
        # the largest source run, primaries and tallies kept on the device
        {"name": "source_1e6_fp64", "kind": "source", "n": 1_000_000, "nz": 1000, "column": 5e21,
         "length": 10.0, "precision": FP64, "device": True},
        # precision form of a thinner source with an odd size and segmentation
        {"name": "source_3e5_fp32", "kind": "source", "n": 299_993, "nz": 777, "column": 3.1e21,
         "length": 7.3, "precision": FP32, "device": True},
        # continuous field update: the run in four cycles of a quarter each
        {"name": "cycles_5e4_fp64", "kind": "cycles", "n": 50_000, "nz": 1000, "column": 5e21,
         "length": 10.0, "cycles": 4, "precision": FP64},
        # source with T+ from dissociative ionization, three-body clustering
        # and charge exchange
        {"name": "chemistry_3e3_fp64", "kind": "chemistry", "n": 3000, "nz": 100,
         "column": 2e21, "length": 4.0, "precision": FP64},
        # thermalisation check: every collision on a moving target
        {"name": "thermal_2e3_fp64", "kind": "thermal", "n": 2000, "density": 3e21,
         "precision": FP64},
        # a parameter scan: uneven source configurations in one server launch
        {"name": "batch_16_fp32", "kind": "batch", "n": 16, "lo": 1e3, "hi": 3e4, "nz": 1000,
         "precision": FP32},
        # ions in the tube at the full field, gyration resolved
        {"name": "orbit_ions_32k", "kind": "orbit_ions", "n": 32768, "lifetime": 3e-5},
        # beta electrons, ions and their products in the tube
        {"name": "orbit_tube_300", "kind": "orbit_tube", "n": 300, "lifetime": 1e-7},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["thin", "source", "source", "source", "cycles", "chemistry", "thermal",
                       "batch", "orbit_ions", "orbit_tube"])
    prec = rng.choice([FP64, FP32])
    if kind == "thin":
        return {"kind": kind, "n": _log_int(rng, 1e3, 1e5), "nz": rng.randint(100, 1200),
                "precision": prec, "angular": rng.random() < 0.5}
    col, length = rng.uniform(0.1, 1.0) * 5e21, rng.uniform(2.0, 10.0)
    nz = rng.randint(100, 1200)
    if kind == "source":
        return {"kind": kind, "n": _log_int(rng, 1e3, 1e6), "nz": nz, "column": col,
                "length": length, "precision": prec, "device": rng.random() < 0.5}
    if kind == "cycles":
        return {"kind": kind, "n": _log_int(rng, 1e3, 1e5), "nz": nz, "column": col,
                "length": length, "cycles": rng.randint(2, 8), "precision": prec}
    if kind == "chemistry":
        return {"kind": kind, "n": _log_int(rng, 1e3, 3e4), "nz": rng.randint(50, 400),
                "column": rng.uniform(0.5, 1.0) * 2e21, "length": rng.uniform(2.0, 6.0),
                "precision": prec}
    if kind == "thermal":
        return {"kind": kind, "n": _log_int(rng, 200, 5000), "density": _log(rng, 5e20, 3e21),
                "precision": prec}
    if kind == "batch":
        return {"kind": kind, "n": rng.randint(4, 24), "lo": 1e3, "hi": _log(rng, 3e3, 3e4),
                "nz": rng.randint(400, 1100), "precision": prec}
    if kind == "orbit_ions":
        return {"kind": kind, "n": _log_int(rng, 1e3, 131072), "lifetime": _log(rng, 3e-6, 3e-5)}
    return {"kind": kind, "n": _log_int(rng, 50, 2000), "lifetime": _log(rng, 2e-8, 1e-7)}


# ---------------------------------------------------------------------------
# preparation

def _problem(case, seed):
    k, n = case["kind"], case["n"]
    if k == "thin":
        prob, prims = inputs.config1(n, seed, nz=case["nz"])
        if case["angular"]:
            prob.channels[0].angular = inputs.screened_rutherford_table()
        return prob, prims
    if k in ("source", "cycles"):
        return inputs.config2(n, seed, column_m2=case["column"], length=case["length"],
                              nz=case["nz"])
    if k == "chemistry":
        return inputs.chemistry_config(n, seed, column_m2=case["column"], length=case["length"],
                                       nz=case["nz"])
    return inputs.thermalization(n, seed, density_m3=case["density"])


def _device_buffers(prob, prims):
    dev = torch.device("cuda", torch.cuda.current_device())
    src = {k: torch.from_numpy(np.ascontiguousarray(getattr(prims, k))).to(dev)
           for k in ("z_m", "e_ev", "mu", "species")}
    nz, ntb, ns = prob.n_zbins, prob.n_tebins, karl.N_SPECIES
    i64, f64 = torch.int64, torch.float64
    shapes = {"spectrum": ((2, ns, prob.n_spec_bins + 1), i64), "time_fx": ((ns, nz + 2, ntb), i64),
              "cross_pos": ((ns, nz + 1), i64), "cross_neg": ((ns, nz + 1), i64),
              "recomb": ((ns, nz), i64), "ledger": ((karl.LEDGER_LEN,), i64),
              "chan_count": ((prob.n_channels,), i64), "per_primary": ((prims.n,), i64),
              "density": ((ns, nz), f64), "current": ((ns, nz + 1), f64),
              "field": ((ns, nz, ntb), f64)}
    out = {k: torch.zeros(s, dtype=t, device=dev) for k, (s, t) in shapes.items()}
    torch.cuda.synchronize()
    return src, out


def prepare(case, seed):
    seed = int(seed) % (1 << 31) + 1
    k = case["kind"]
    torch.cuda.init()
    st = {"case": case, "seed": seed}
    if k == "batch":
        batch = inputs.config4_batch(case["n"], seed, case["lo"], case["hi"], nz=case["nz"])
        st["batch"] = batch
        st["server"] = karl.Server(batch[0][0], precision=case["precision"], max_slots=64,
                                   hbm_budget_bytes=2 << 30)
        return st
    if k == "orbit_ions":
        prob, st["orbit"], st["prims"] = inputs.orbit_ion_config(case["n"], seed,
                                                                 lifetime_s=case["lifetime"])
    elif k == "orbit_tube":
        prob, st["orbit"], st["prims"] = inputs.orbit_config(case["n"], seed,
                                                             lifetime_s=case["lifetime"])
    else:
        prob, prims = _problem(case, seed)
        st["prims"] = prims
        if k == "source" and case["device"]:
            st["src"], st["out"] = _device_buffers(prob, prims)
    st["ctx"] = karl.Context(prob)
    return st


# ---------------------------------------------------------------------------
# one call

def _signed(tallies):
    """The tallies with counts as signed 64-bit views (torch and most file
    formats take no unsigned 64-bit values)."""
    return {k: v.view(np.int64) if v.dtype == np.uint64 else v for k, v in tallies.items()}


def run(st):
    case, seed = st["case"], st["seed"]
    k = case["kind"]
    if k == "batch":
        srv = st["server"]
        ids = [srv.submit(p, q, s) for p, q, s in st["batch"]]
        srv.run_all()
        done = [srv.poll(i)[1] for i in ids]
        # a scan's results by tally, one row per configuration
        return _signed({key: np.stack([t[key] for t in done]) for key in done[0]})
    ctx, prims = st["ctx"], st["prims"]
    if k in ("orbit_ions", "orbit_tube"):
        return _signed(ctx.run_orbit(st["orbit"], prims, seed=seed))
    if k == "cycles":
        return _signed(ctx.run_cycles(prims, seed, case["cycles"], precision=case["precision"]))
    if k == "source" and case["device"]:
        ctx.run_device({n: t.data_ptr() for n, t in st["src"].items()}, prims.n, prims.n_decays,
                       {n: t.data_ptr() for n, t in st["out"].items()}, seed=seed,
                       precision=case["precision"])
        return st["out"]
    return _signed(ctx.run(prims, seed=seed, precision=case["precision"]))


# ---------------------------------------------------------------------------
# what a call cannot do without

# floating-point operations of one collision (flight, channel choice, elastic
# kinematics) and of one Boris step, counted from the formulas with a root,
# a logarithm, a cosine and a division as one operation each
OPS_COLLISION, OPS_STEP = 60.0, 85.0


def work(case):
    k, n = case["kind"], case["n"]
    nz, ntb = case.get("nz", 200), 1 if k in ("thin", "thermal") else 64
    spec = 2 * 4 * 20001 * 8
    tallies = spec + 4 * (nz + 2) * ntb * 8 + 4 * nz * ntb * 8 + 2 * 4 * (nz + 1) * 8 + \
        2 * 4 * nz * 8 + 4 * (nz + 1) * 8
    if k == "thin":
        return {"bytes": n * (25 + 8) + tallies, "flops": n * 3.8 * OPS_COLLISION}
    if k in ("source", "cycles", "chemistry"):
        passes = 1 if k == "cycles" else 2
        # collisions per decay grow a little more than linearly with the column
        coll = 1660.0 * min(1.0, case["column"] / 5e21)
        return {"bytes": 2 * n * (25 + 8) + tallies, "flops": passes * n * coll * OPS_COLLISION}
    if k == "thermal":
        # random walk from the middle: about (n sigma L / 2)^2 / 0.66 collisions
        mfp = case["density"] * 1e-19 * 0.1
        return {"bytes": n * (25 + 8) + tallies, "flops": n * 1.5 * mfp * mfp * OPS_COLLISION}
    if k == "batch":
        decays = n * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": 2 * decays * 25 + n * tallies,
                "flops": 2 * decays * 0.55 * 1660.0 * OPS_COLLISION}
    if k == "orbit_ions":
        dt = float(inputs.boris_dt(2.5)[inputs.T2P])
        steps = n * 1.1 * case["lifetime"] / dt
    else:
        dt = float(inputs.boris_dt(0.25)[inputs.E])
        steps = n * 0.6 * case["lifetime"] / dt
    return {"bytes": n * (49 + 8 + 64), "flops": steps * OPS_STEP}


# ---------------------------------------------------------------------------
# the thin-column workloads in numpy, 64 bits

_U = np.uint64


def _mulhilo(a, b):
    m32, s32 = _U(0xFFFFFFFF), _U(32)
    al, ah, bl, bh = a & m32, a >> s32, b & m32, b >> s32
    ll, lh, hl = al * bl, al * bh, ah * bl
    mid = (ll >> s32) + (lh & m32) + (hl & m32)
    return ah * bh + (lh >> s32) + (hl >> s32) + (mid >> s32), a * b


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x64-10 (Salmon et al., SC'11)."""
    m0, m1 = _U(0xD2E7470EE14C6C93), _U(0xCA5A826395121157)
    w0, w1 = _U(0x9E3779B97F4A7C15), _U(0xBB67AE8584CAA73B)
    for _ in range(10):
        h0, l0 = _mulhilo(np.broadcast_to(m0, c0.shape), c0)
        h1, l1 = _mulhilo(np.broadcast_to(m1, c2.shape), c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = k0 + w0, k1 + w1
    return c0, c1, c2, c3


def _mix(x):
    z = x + _U(0x9E3779B97F4A7C15)
    z = (z ^ (z >> _U(30))) * _U(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> _U(27))) * _U(0x94D049BB133111EB)
    return z ^ (z >> _U(31))


def _table_cchi(tab, e, u):
    """cos(chi) from a pdf linear between even points, by its cumulative integral."""
    nb, n = tab.pdf.shape
    h = 2.0 / (n - 1)
    cum = np.concatenate([np.zeros((nb, 1)),
                          np.cumsum(0.5 * h * (tab.pdf[:, 1:] + tab.pdf[:, :-1]), axis=1)], axis=1)
    b = np.floor(nb * np.log(e / tab.e_min_ev) / math.log(tab.e_max_ev / tab.e_min_ev))
    b = np.clip(b.astype(int), 0, nb - 1)
    t = u * cum[b, -1]
    lo, hi = np.zeros(len(e), int), np.full(len(e), n - 1)
    while np.any(hi - lo > 1):
        mid = (lo + hi) >> 1
        left = cum[b, mid] <= t
        lo, hi = np.where(left, mid, lo), np.where(left, hi, mid)
    r, a = t - cum[b, lo], tab.pdf[b, lo]
    s = (tab.pdf[b, lo + 1] - a) / h
    den = a + np.sqrt(np.maximum(0.0, a * a + 2 * s * r))
    return np.minimum(1.0, -1 + lo * h + np.clip(2 * r / np.where(den > 0, den, 1.0), 0, h))


def exact(case, seed):
    if case["kind"] != "thin":
        return None                # 1e6 to 1e9 collisions or steps
    with np.errstate(over="ignore"):
        return _thin_exact(case, int(seed) % (1 << 31) + 1)


def _thin_exact(case, seed):
    prob, pr = _problem(case, seed)
    Q, QT, c = 2.0 ** 24, 2.0 ** 50, 299792458.0
    nz, length = prob.n_zbins, prob.length_m
    dz = length / nz
    dens = float(prob.n_seg_m3[0])
    m = float(prob.species_mass_ev[0])
    g = m / prob.target_mass_ev
    sig, loss = prob.sigma_matrix(), np.array([ch.loss_ev for ch in prob.channels])
    loss_q = np.floor(loss * Q).astype(np.int64)
    h = math.log(prob.e_max_ev / prob.e_min_ev) / (prob.n_energy - 1)
    ecut = int(math.floor(prob.e_cut_ev * Q))
    tpt, trg = np.zeros(nz + 3), np.zeros(nz + 3)
    cross = np.zeros((2, nz + 3))
    z, mu = pr.z_m.copy(), pr.mu.copy()
    eq = np.floor(pr.e_ev * Q).astype(np.int64)
    pid = np.arange(pr.n, dtype=_U)
    node, ev = np.zeros(pr.n, _U), np.zeros(pr.n, np.int64)
    keep = eq >= ecut
    z, mu, eq, pid, node, ev = (a[keep] for a in (z, mu, eq, pid, node, ev))
    while len(z):
        e = eq / Q
        zero = np.zeros(len(z), _U)
        w = _philox(ev.astype(_U), node, zero + _U(1 << 8), zero, zero + _U(seed), pid)
        u = [(x >> _U(11)).astype(np.float64) * 2.0 ** -53 for x in w]
        tau = -np.log(((w[0] >> _U(11)) + _U(1)).astype(np.float64) * 2.0 ** -53)
        lx = np.log(e / prob.e_min_ev) / h
        i = np.clip(np.floor(lx).astype(int), 0, prob.n_energy - 2)
        f = np.clip(lx - i, 0.0, 1.0)
        s = np.where(eq[None, :] > loss_q[:, None],
                     sig[:, i] + f * (sig[:, i + 1] - sig[:, i]), 0.0)
        gas = s.sum(axis=0)
        up = mu > 0
        znew = z + np.where(up, 1.0, -1.0) * tau * np.abs(mu) / (gas * dens)
        out = (znew >= length) | (znew <= 0.0)
        znew = np.clip(znew, 0.0, length)
        x = e / m
        per_m = (1 + x) / np.sqrt(x * (2 + x)) / c / np.abs(mu)      # seconds per metre along z
        j0 = np.clip(np.floor(z / dz).astype(int), 0, nz - 1)
        j1 = np.clip(np.floor(znew / dz).astype(int), 0, nz - 1)
        same = j0 == j1
        first = np.abs(np.where(same, znew, np.where(up, j0 + 1, j0) * dz) - z)
        last = np.where(out, dz, np.abs(znew - np.where(up, j1, j1 + 1) * dz))
        q = lambda d: np.floor(d * per_m * QT + 0.5)                 # units of 2^-50 s
        np.add.at(tpt, j0, q(first))
        np.add.at(tpt, j1[~same], q(last)[~same])
        a, b = np.minimum(j0, j1) + 1, np.maximum(j0, j1)
        np.add.at(trg, a[~same], q(dz)[~same])
        np.add.at(trg, b[~same], -q(dz)[~same])
        fa = np.where(up, j0 + 1, np.where(out, 0, j1 + 1))
        fb = np.where(up, np.where(out, nz, j1), j0) + 1
        for way, sel in ((0, up & (fb > fa)), (1, ~up & (fb > fa))):
            np.add.at(cross[way], fa[sel], 1)
            np.add.at(cross[way], fb[sel], -1)
        # collisions
        k = ~out
        z, mu, eq, pid, node, ev, e = (a[k] for a in (znew, mu, eq, pid, node, ev, e))
        s, gas, u = s[:, k], gas[k], [x[k] for x in u]
        ch = np.argmax(u[1] * gas < np.cumsum(s, axis=0), axis=0)
        cphi = np.cos(2 * math.pi * u[3])
        smu = np.sqrt(np.maximum(0.0, 1 - mu * mu))
        el, io = ch == 0, ch == 1
        # elastic
        cchi = 2 * u[2] - 1
        tab = prob.channels[0].angular
        if tab is not None:
            hi = el & (e >= tab.threshold_ev)
            cchi[hi] = _table_cchi(tab, e[hi], u[2][hi])
        ct = (cchi + g) / np.sqrt(1 + 2 * g * cchi + g * g)
        de = np.floor(e * 2 * g * (1 - cchi) / (1 + g) ** 2 * Q + 0.5).astype(np.int64)
        mu_el = mu * ct + smu * np.sqrt(np.maximum(0.0, 1 - ct * ct)) * cphi
        # ionization: energy sharing and binary-encounter angles
        avail = np.maximum(eq - loss_q[1], 1)
        eps = prob.ioniz_eps_ev
        wsec = eps * np.tan(u[2] * np.arctan(0.5 * np.maximum(e - loss[1], 0.0) / eps))
        wq = np.clip(np.floor(wsec * Q).astype(np.int64), 0, avail // 2)
        cp, sp = np.sqrt((avail - wq) / avail), np.sqrt(wq / avail)
        born = io & (wq >= ecut)
        new = (z[born], np.clip(mu * sp - smu * cp * cphi, -1, 1)[born], wq[born], pid[born],
               _mix(_mix(node) ^ (ev.astype(_U) << _U(2)))[born], np.zeros(int(born.sum()), np.int64))
        eq = np.where(el, eq - de, np.where(io, avail - wq, eq - loss_q[ch]))
        mu = np.where(el, np.clip(mu_el, -1, 1),
                      np.where(io, np.clip(mu * cp + smu * sp * cphi, -1, 1), mu))
        keep = eq >= ecut
        z, mu, eq, pid, node, ev = (np.concatenate([a[keep], b]) for a, b in
                                    zip((z, mu, eq, pid, node, ev + 1), new))
    t = (tpt + np.cumsum(trg))[:nz] / QT
    tsim = pr.n_decays / prob.activity_bq
    vol = dz * prob.area_m2
    density, current = np.zeros((4, nz)), np.zeros((4, nz + 1))
    density[0] = t / (tsim * vol)
    way = np.cumsum(cross, axis=1)[:, :nz + 1]
    current[0] = (way[0] - way[1]) / (prob.area_m2 * tsim)
    none = dict.fromkeys(("spectrum", "time_fx", "cross_pos", "cross_neg", "recomb", "ledger",
                          "chan_count", "per_primary"))
    return {**none, "density": density, "current": current,
            "field": density.reshape(4, nz, 1).copy()}
