"""Timed cases of the fragment kMC library: what a user's program does between
creating a batch and reading its results.

Each case builds a batch of lattices (sizes, compositions, barriers and options
of the workloads in ``paper_2004_09081_gb300.workloads``, or smaller and larger
ones of the same kind), and one pass advances it by a number of windows (or
null-event steps, or solves its potential) and reads the results a simulation
keeps: hop counts, displacement moments, and the vacancy records, ion positions
and tracer field where the lattice is of a size that is read back whole.  A pass
continues from the state the last one left, as a sampling loop does.
"""
from __future__ import annotations

import math

import numpy as np

from paper_2004_09081_gb300 import fkmc, workloads
from paper_2004_09081_gb300.workloads import A_BATIO3, A_SRTIO3, Replica, round_half_up

# Fields of a lattice case (every replica has the same cells; T runs evenly from
# T to T_hi over the replicas): replicas, nx, ny, nz, a (Angstrom), f_vac
# (vacancies per O site), x_H (H- per cell), f_fe (dopants per cell), T, T_hi,
# Ea_O, Ea_H, field (V/m along z), edge (fragment edge, cells), n_tau, precision
# ("plain" FP64 or "mixed" integer rates), tracer, windows or steps per pass, and
# the optional parts: site (interaction energies), grains (Voronoi seeds),
# eps_r (electrostatics), cap_v (vacancy slots per fragment, 0: sized from the
# composition).  read: what a pass reads back besides the counts and moments.
_LATTICE = dict(kind="windows", replicas=1, f_vac=0.001, x_H=0.0, f_fe=0.0, field=0.0, edge=4, n_tau=0.5,
                precision="plain", tracer=False, site=False, grains=0, eps_r=0.0, cap_v=0, read="records")
_STO = dict(a=A_SRTIO3, Ea_O=0.60, Ea_H=0.60)
_BTO = dict(a=A_BATIO3, Ea_O=0.70, Ea_H=0.35)


def _lattice(cells, **kw):
    nx, ny, nz = (cells,) * 3 if isinstance(cells, int) else cells
    c = dict(_LATTICE, nx=nx, ny=ny, nz=nz)
    c.update(kw)
    c.setdefault("T_hi", c["T"])
    return c


def listed():
    return [
        # the smallest call: one 8^3 SrTiO3 cell block, 15 vacancies, FP64 (the default form),
        # a few windows between readings
        _lattice(8, name="small_plain_8c", f_vac=15 / 1536, T=800.0, windows=16, **_STO),
        # temperature sweep of hydride SrTiO3 in the plain form with every ion traced
        _lattice(32, name="sweep_plain_5x32c", replicas=5, f_vac=0.005, x_H=0.1, T=300.0, T_hi=700.0, tracer=True,
                 windows=400, read="records,state,tracer", **dict(_STO, Ea_H=0.30)),
        # the uneven batch of BaTiO(3-x)H_x replicas that the benchmark runs (16..48 cells, mixed form)
        dict(name="batch_mixed_256", kind="batch", replicas=256, batch_seed=0, edge=5, n_tau=0.5, windows=3072,
             read="records"),
        # the paper's hydride runs: two materials x three concentrations x four temperatures, traced
        dict(name="trend_mixed_24x32c", kind="trend", L=32, windows=8000, read="records,tracer"),
        # one lattice too large for an SM, both arithmetic forms; positions of every ion read back
        _lattice(128, name="bulk_mixed_128c", f_vac=0.003, x_H=0.05, T=400.0, edge=8, precision="mixed",
                 windows=2000, read="records,state", **_BTO),
        _lattice(128, name="bulk_plain_128c", f_vac=0.003, x_H=0.05, T=400.0, edge=8, windows=1000,
                 read="records,state", **_BTO),
        # dopant and vacancy interactions over a temperature range
        _lattice(96, name="dopant_plain_5x96c", replicas=5, f_fe=0.001, T=600.0, T_hi=1000.0, site=True, windows=512,
                 **_STO),
        # vacancies in their own potential, solved again every eight windows, under bias
        _lattice(128, name="elec_plain_128c", T=400.0, field=1e7, eps_r=1000.0, windows=64, **dict(_BTO, Ea_H=0.70)),
        # the potential alone, as a map of the sample's state
        _lattice(128, name="potential_128c", kind="potential", T=400.0, eps_r=1000.0, cycles=12, read="",
                 **dict(_BTO, Ea_H=0.70)),
        # the atom-based form with null events, one pick per vacancy and step
        _lattice(128, name="null_128c", kind="null", f_vac=0.003, x_H=0.05, T=400.0, edge=8, precision="mixed",
                 steps=2000, read="records,state", **_BTO),
        # grains in a box of the paper's proportions (1600 x 400 x 2400 cells at half the edge); vacancies
        # gather at the boundary layers under the bias, hence the larger capacity per fragment
        _lattice((800, 200, 1200), name="grains_mixed_192M", T=400.0, field=2.08e7, edge=8, precision="mixed",
                 grains=16, cap_v=64, windows=100, read="", **dict(_BTO, Ea_H=0.70)),
        # the mu-scale cube under bias: too large to read back, only drift and diffusion are kept
        _lattice(1300, name="um_mixed_1300c", T=400.0, field=1e7, edge=8, precision="mixed", windows=80, read="",
                 **dict(_BTO, Ea_H=0.70)),
    ]


def _log_int(rng, lo, hi):
    return round_half_up(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    """A case of the listed ranges: lattice edges, compositions, temperatures,
    fragment edges, window lengths and pass lengths vary, the kinds are those
    above."""
    kind = rng.choice(["small", "sweep", "batch", "trend", "bulk", "dopant", "elec", "potential", "null", "grains",
                       "um"])
    n_tau = rng.choice([0.25, 0.5, 1.0])
    prec = rng.choice(["plain", "mixed"])
    if kind == "small":
        L = rng.randint(8, 24)
        return _lattice(L, f_vac=rng.uniform(0.002, 0.01), T=rng.uniform(300.0, 1000.0), edge=rng.randint(4, 6),
                        n_tau=n_tau, precision=prec, windows=_log_int(rng, 4, 256), **_STO)
    if kind == "sweep":
        L = rng.randint(20, 40)
        return _lattice(L, replicas=rng.randint(2, 8), f_vac=rng.uniform(0.001, 0.008), x_H=rng.uniform(0.02, 0.3),
                        T=300.0, T_hi=rng.uniform(500.0, 900.0), tracer=True, n_tau=n_tau, precision=prec,
                        windows=_log_int(rng, 50, 500), read="records,state,tracer", **dict(_STO, Ea_H=0.30))
    if kind == "batch":
        return dict(kind="batch", replicas=_log_int(rng, 16, 256), batch_seed=rng.randint(1, 10 ** 6),
                    edge=rng.randint(5, 8), n_tau=rng.choice([0.25, 0.5]), windows=_log_int(rng, 256, 2048),
                    read="records")
    if kind == "trend":
        return dict(kind="trend", L=rng.randint(24, 34), windows=_log_int(rng, 500, 6000), read="records,tracer")
    if kind == "bulk":
        L = rng.randint(64, 128)
        return _lattice(L, f_vac=rng.uniform(0.001, 0.003), x_H=rng.uniform(0.0, 0.15), T=rng.uniform(350.0, 700.0),
                        edge=rng.randint(6, 8), n_tau=n_tau, precision=prec, windows=_log_int(rng, 100, 1000),
                        read="records,state", **_BTO)
    if kind == "dopant":
        L = 8 * rng.randint(4, 12)
        return _lattice(L, replicas=rng.randint(1, 5), f_vac=rng.uniform(0.0005, 0.002),
                        f_fe=rng.uniform(0.0005, 0.002), T=rng.uniform(500.0, 700.0), T_hi=rng.uniform(800.0, 1000.0),
                        n_tau=n_tau, site=True, windows=_log_int(rng, 32, 512), **_STO)
    if kind == "elec":
        L = 8 * rng.randint(6, 16)
        return _lattice(L, T=rng.uniform(350.0, 700.0), field=1e7, eps_r=rng.uniform(300.0, 2000.0),
                        n_tau=n_tau, windows=_log_int(rng, 16, 64), **dict(_BTO, Ea_H=0.70))
    if kind == "potential":
        nx, ny, nz = (4 * rng.randint(8, 32) for _ in range(3))
        return _lattice((nx, ny, nz), kind="potential", T=400.0, eps_r=rng.uniform(300.0, 2000.0), cycles=12,
                        read="", **dict(_BTO, Ea_H=0.70))
    if kind == "null":
        L = rng.randint(32, 128)
        return _lattice(L, kind="null", f_vac=rng.uniform(0.001, 0.004), x_H=rng.uniform(0.0, 0.15), T=400.0, edge=8,
                        precision=prec, steps=_log_int(rng, 100, 1500), read="records,state", **_BTO)
    if kind == "grains":
        cells = (8 * rng.randint(30, 100), 8 * rng.randint(20, 25), 8 * rng.randint(40, 150))
        return _lattice(cells, T=rng.uniform(350.0, 600.0), field=1e7, edge=8, n_tau=n_tau, precision="mixed",
                        grains=rng.randint(4, 16), cap_v=64, windows=_log_int(rng, 20, 100), read="",
                        **dict(_BTO, Ea_H=0.70))
    L = rng.randint(520, 1300)
    return _lattice(L, f_vac=rng.uniform(0.0005, 0.001), T=rng.uniform(350.0, 600.0), field=1e7, edge=rng.randint(6, 8),
                    precision="mixed", windows=_log_int(rng, 10, 60), read="", **dict(_BTO, Ea_H=0.70))


def _replicas(c):
    if c["kind"] == "batch":
        return workloads.batched_batio3(c["batch_seed"], c["replicas"]).replicas
    if c["kind"] == "trend":
        return workloads.h_trend(0, c["L"]).replicas
    ncell = c["nx"] * c["ny"] * c["nz"]
    n_vac = max(1, round_half_up(c["f_vac"] * 3 * ncell))
    n = c["replicas"]
    return [Replica((c["nx"], c["ny"], c["nz"]), c["a"], n_vac, round_half_up(c["x_H"] * ncell),
                    c["T"] + (c["T_hi"] - c["T"]) * (r / (n - 1) if n > 1 else 0.0), c["Ea_O"], c["Ea_H"], c["field"],
                    n_Fe=round_half_up(c["f_fe"] * ncell)) for r in range(n)]


def _options(c):
    if c["kind"] == "batch":
        return dict(edge=c["edge"], n_tau=c["n_tau"], precision=fkmc.FKMC_MIXED, schedule=0, cluster_top=0)
    if c["kind"] == "trend":
        return dict(edge=4, n_tau=0.5, precision=fkmc.FKMC_MIXED, tracer=True)
    return dict(edge=c["edge"], n_tau=c["n_tau"], tracer=c["tracer"], cap_v=c["cap_v"],
                precision=fkmc.FKMC_MIXED if c["precision"] == "mixed" else fkmc.FKMC_PLAIN)


def _occupancy(case, seed):
    """Vacancies of the potential case, placed at random: one species code per site."""
    nsite = 3 * case["nx"] * case["ny"] * case["nz"]
    g = np.random.Generator(np.random.Philox(key=np.array([seed, 0x90B0], np.uint64)))
    occ = np.zeros(nsite, np.uint8)
    occ[g.choice(nsite, _replicas(case)[0].n_vac, replace=False, shuffle=False)] = fkmc.FKMC_V
    return occ


def prepare(case, seed):
    reps = _replicas(case)
    b = fkmc.Batch([(*r.cells, r.a) for r in reps], [(r.n_vac, r.n_H, r.n_Fe) for r in reps], seed=seed,
                   **_options(case))
    b.set_barriers([r.Ea_O for r in reps], [r.Ea_H for r in reps], [r.T for r in reps],
                   field_z=[r.field_z for r in reps])
    if case.get("grains"):
        b.set_grains(case["grains"], 1, 0.2)
    if case.get("site"):
        b.set_site_energy(workloads.PAPER_VV, workloads.PAPER_VFE)
    if case["kind"] == "potential":
        b.write_state(_occupancy(case, seed))
        b.set_electrostatics(case["eps_r"], 2.0, refresh_windows=0, cycles=case["cycles"])
    elif case.get("eps_r"):
        b.set_electrostatics(case["eps_r"], 2.0, refresh_windows=8, cycles=12, warm_cycles=6)
    return case, b


def run(state):
    case, b = state
    if case["kind"] == "potential":
        phi, _ = b.solve_potential()
        return phi
    if case["kind"] == "null":
        s = b.run_null(case["steps"], max(c.n_vac for c in b.comps))
    else:
        s = b.run(case["windows"])
    out = {"hops": int(s.hops), "handoffs": int(s.handoffs), "moments": b.moments_all()}
    read = case["read"].split(",")
    if "records" in read:
        out["records"] = np.concatenate([b.records(r) for r in range(b.n)])
    if "state" in read:
        out["state"] = np.concatenate([b.state(r) for r in range(b.n)])
    if "tracer" in read:
        out["tracer"] = np.concatenate([b.tracer_field(r) for r in range(b.n)])
    return out


def _hops(case, r):
    """Expected exchanges of one pass of one replica: a vacancy hops with the mean
    rate of its neighbours' species, a window lasts n_tau / (8 k_fast)."""
    nsite = 3.0 * r.cells[0] * r.cells[1] * r.cells[2]
    kT = 8.617333262e-5 * r.T
    k_O, k_H = math.exp(-r.Ea_O / kT), math.exp(-r.Ea_H / kT)
    p_H = r.n_H / nsite
    mean = (1.0 - p_H) * k_O + p_H * k_H
    if case["kind"] == "null":  # picks of a step that are not null: mean total over the largest
        return r.n_vac * case["steps"] * mean / (k_H if r.n_H else k_O)
    n_tau = case.get("n_tau", 0.5)
    return r.n_vac * case["windows"] * n_tau * mean / (max(k_O, k_H) if r.n_H else k_O)


def work(case):
    """Bytes: the state read and written once (2 bits per site, 24 bytes per vacancy,
    12 per traced site), 160 per exchange (8 neighbour sectors, two sites, a record),
    the outputs; the null-event form also reads every vacancy and its neighbours once
    per step (56 bytes) and its picks' claims.  Operations: 10 Philox rounds of 8
    multiplies and the selection per exchange."""
    if case["kind"] == "potential":
        n = case["nx"] * case["ny"] * case["nz"]
        # deposit and potential once; per cycle the FP64 defect and update, the FP32 smoothing
        # of every level (8/7 of the finest): one read and one write of the potential
        return {"bytes": 8.0 * n + 16.0 * n * case["cycles"], "flops": case["cycles"] * n * (10.0 + 4 * 8.0 * 8 / 7)}
    b = f = 0.0
    for r in _replicas(case):
        nsite = 3.0 * r.cells[0] * r.cells[1] * r.cells[2]
        hops = _hops(case, r)
        b += 2 * (nsite / 4 + 24.0 * r.n_vac) + 160.0 * hops
        f += 120.0 * hops
        if case.get("tracer") or case["kind"] == "trend":
            b += 24.0 * hops
        if case["kind"] == "null":
            b += 56.0 * r.n_vac * case["steps"]
            f += 120.0 * r.n_vac * case["steps"]
        if case.get("site"):
            b += 964.0 * hops  # the moved vacancy's shells of the energy field
        if case.get("eps_r"):
            n = nsite / 3
            b += case["windows"] / 8 * (6 * 16.0 * n + 24.0 * n)
            f += case["windows"] / 8 * 6 * n * (10.0 + 4 * 8.0 * 8 / 7)
        read = case["read"].split(",")
        b += (48.0 * r.n_vac if "records" in read else 0.0) + (nsite if "state" in read else 0.0)
        b += 12.0 * nsite if "tracer" in read else 0.0
    return {"bytes": b, "flops": f}


def exact(case, seed):
    """The potential from the discrete equation solved by a Fourier transform; the
    trajectories are whole numbers."""
    if case["kind"] != "potential":
        return None
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    vac = (_occupancy(case, seed) == fkmc.FKMC_V).reshape(3, nz, ny, nx)
    half = np.zeros((nz, ny, nx))
    for t in range(3):  # half a charge on each end of the site's bond
        half += vac[t]
        half += np.roll(vac[t], 1, axis=2 - t)
    scale = 1.602176634e-19 / (8.8541878128e-12 * case["eps_r"] * case["a"] * 1e-10)
    f = (2.0 / 2 * half - 2.0 * vac.sum() / half.size) * scale
    k = [2.0 - 2.0 * np.cos(2.0 * np.pi * np.arange(n) / n) for n in (nz, ny, nx)]
    lam = k[0][:, None, None] + k[1][None, :, None] + k[2][None, None, :]
    F = np.fft.fftn(f)
    lam[0, 0, 0] = 1.0
    F /= lam
    F[0, 0, 0] = 0.0
    return np.real(np.fft.ifftn(F)).ravel()
