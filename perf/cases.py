"""Timed cases of the dose engine: what its users call, over the sizes they call it with.

A case names a form of the call, a phantom, a beam and a history count:

* ``simulate``   one dose calculation on a resident phantom, dose and sigma in host arrays
* ``e2e``        the same from a host phantom: upload, simulate, release
* ``plan``       a resident plan from a zeroed tally to dose and sigma on the device
* ``batch``      uneven plans of both particle types in one ``run``, then their results
* ``target``     uneven plans run together until each reaches its uncertainty
* ``served``     requests through ``serve.Server`` until each reaches its uncertainty
* ``readout``    the FP64 dose and sigma of a plan that already holds its histories

The transport is a Monte Carlo whose random streams are keyed by the seed, and
whose tally is an integer sum: the same inputs give the same bits, and no other
program gives them, so ``exact`` has no value to offer for any case.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import workloads as W
import paper_1101_1245_gb300 as g
from paper_1101_1245_gb300 import serve

# What depends on the histories alone, not on how they were scheduled.
COUNTS = ("histories", "e_incident", "e_deposited", "e_escaped", "e_rest", "n_photon_events", "n_photon_real",
          "n_compton", "n_photo", "n_pair", "n_electron_steps", "n_hard_real", "n_hard_fict", "n_moller", "n_brem",
          "n_photons", "n_electrons", "n_sampler_capped")


def _case(name, form, phantom, nx, ny, nz, voxel, particle, energy, field, histories, batches, source="mono",
          plans=1, target=0.0, kerma=False):
    """source: mono, spectrum (6 MV-like photons, flat 1-15 MeV electrons),
    grouped (the spectrum, claimed by energy) or phsp (a grouped phase space)."""
    c = dict(form=form, phantom=phantom, nx=nx, ny=ny, nz=nz, voxel=voxel, particle=particle, energy=energy,
             field=field, histories=histories, batches=batches, source=source, plans=plans, target=target,
             kerma=kerma)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a quick look at a beam: few histories, odd sizes, unequal batches; latency alone
        _case("probe_ragged_e", "simulate", "slabs", 31, 27, 45, 0.4, "electron", 9.0, 3.0, 3001, 32),
        # the smallest configuration: a 2 MeV photon pencil in 32^3 water
        _case("pencil_water32_g", "simulate", "water", 32, 32, 32, 0.5, "photon", 2.0, 0.0, 100_000, 32),
        # the timing configuration of the paper, its two beams
        _case("water128_e", "plan", "water", 128, 128, 128, 0.25, "electron", 15.0, 10.0, 1_000_000, 16),
        _case("water128_g", "plan", "water", 128, 128, 128, 0.25, "photon", 15.0, 10.0, 4_000_000, 16),
        # the slab configuration: a polyenergetic field on a large grid
        _case("slabs256_6mv", "plan", "slabs", 256, 256, 256, 0.2, "photon", 0.0, 10.0, 10_000_000, 16, "spectrum"),
        # a plan as a planning system sends it: CT-like phantom up, dose back, nothing resident
        _case("ct_thorax_e2e_e", "e2e", "ct", 128, 96, 128, 0.25, "electron", 15.0, 10.0, 1_000_000, 32),
        # the batched configuration: uneven plans on density fields, both particle types
        _case("batch12_mixed", "batch", "noise", 64, 64, 160, 0.3, "mixed", 12.0, 8.0, 800_000, 16, plans=12),
        # plans run to an uncertainty together, the batched configuration's own stopping rule
        _case("target_mixed", "target", "noise", 64, 64, 128, 0.4, "mixed", 12.0, 6.0, 400_000, 16, plans=6,
              target=0.02),
        # the served configuration: requests on resident phantoms, retired at their uncertainty
        _case("served_mixed", "served", "noise", 64, 64, 112, 0.4, "mixed", 12.0, 6.0, 200_000, 16, plans=8,
              target=0.03),
        # a scored phase space claimed by energy
        _case("phsp_grouped_e", "plan", "water", 128, 128, 128, 0.25, "electron", 0.0, 8.0, 1_000_000, 16, "phsp"),
        # the photon-only fast mode, on the slabs of the paper's third geometry
        _case("kerma_slabs_g", "plan", "slabs", 128, 128, 128, 0.25, "photon", 15.0, 10.0, 4_000_000, 16,
              kerma=True),
        # what every checkpoint of a large plan pays: the fold of its batch tallies
        _case("readout256", "readout", "noise", 256, 256, 256, 0.2, "electron", 12.0, 12.0, 1_000_000, 16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    form = rng.choice(["simulate", "simulate", "plan", "plan", "plan", "e2e", "batch", "target", "served", "readout"])
    many = form in ("batch", "target", "served")
    phantom = "noise" if many else rng.choice(["water", "slabs", "noise", "ct"])
    particle = "mixed" if many else rng.choice(["electron", "photon"])
    top = 128 if form in ("target", "served") else 160 if form == "batch" else 256
    nx, ny, nz = (int(round(_log(rng, 48 if many else 24, top))) for _ in range(3))
    voxel = round(rng.uniform(0.2, 0.5), 3)
    energy = round(rng.uniform(6.0, 18.0), 2)
    field = round(min(_log(rng, 2.0, 15.0), 0.8 * voxel * min(nx, ny)), 2)
    batches = rng.choice([8, 16, 32, 64]) if form in ("plan", "readout") else 16 if many else 32
    if form == "readout":
        return _case(None, form, phantom, nx, ny, nz, voxel, particle, energy, field, int(_log(rng, 1e5, 1e6)), batches)
    if form == "batch":
        return _case(None, form, phantom, nx, ny, nz, voxel, particle, energy, field, int(_log(rng, 5e4, 8e5)),
                     batches, plans=rng.randint(3, 12))
    if form in ("target", "served"):
        return _case(None, form, phantom, nx, ny, nz, max(voxel, 0.4), particle, energy, min(field, 6.0),
                     int(_log(rng, 1e5, 4e5)), batches, plans=rng.randint(2, 6),
                     target=round(rng.uniform(0.03, 0.06), 3))
    histories = int(_log(rng, 1e3, 1e6 if particle == "electron" else 4e6))
    source = rng.choice(["mono", "mono", "spectrum", "grouped", "phsp"]) if form == "plan" else "mono"
    kerma = form == "plan" and source == "mono" and particle == "photon" and rng.random() < 0.3
    return _case(None, form, phantom, nx, ny, nz, voxel, particle, energy if source == "mono" else 0.0, field,
                 histories, batches, source, kerma=kerma)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
_engines = {}


def _engine(case):
    """One context per material set and launch, as a program keeps it."""
    key = (case["phantom"] == "ct", bool(case["kerma"]))
    if key not in _engines:
        ctx = g.engine(0, mats=W.MATERIALS_PAPER if key[0] else W.MATERIALS)
        if key[1]:
            ctx.set_launch(flags=g.LAUNCH_KERMA)
        _engines[key] = ctx
    return _engines[key]


def _density_field(nx, ny, nz, voxel, seed):
    """Gaussian noise smoothed over 2 cm, mapped to 0.2-2.0 g/cm^3, lung below 0.6 and bone above 1.4."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device="cuda"))
    for axis, n in enumerate((nz, ny)):
        k = torch.fft.fftfreq(n, device="cuda") * (2.0 * math.pi * 2.0 / voxel)
        f *= torch.exp(-0.5 * k * k).reshape([-1 if a == axis else 1 for a in range(3)])
    k = torch.fft.rfftfreq(nx, device="cuda") * (2.0 * math.pi * 2.0 / voxel)
    sm = torch.fft.irfftn(f * torch.exp(-0.5 * k * k), s=(nz, ny, nx))
    lo, hi = sm.min(), sm.max()
    rho = (0.2 + (sm - lo) * (1.8 / (hi - lo).clamp_min(1e-30))).float()
    mat = torch.full(rho.shape, W.MAT_WATER, dtype=torch.uint8, device="cuda")
    mat[rho < 0.6] = W.MAT_LUNG
    mat[rho > 1.4] = W.MAT_BONE
    return mat, rho


def _phantom(case, dims, seed):
    """A host phantom of the case's kind; the seed moves its densities within a percent or so."""
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    if case["phantom"] == "ct":
        return W.hu_to_phantom(W.synthetic_ct_hu(dims, case["voxel"], seed), case["voxel"])
    if case["phantom"] == "slabs":
        return W.z_slabs(dims, case["voxel"], [(3.0, W.MAT_WATER, 1.0), (2.0, W.MAT_BONE, 1.85),
                                               (6.0, W.MAT_LUNG, round(rng.uniform(0.25, 0.27), 4)),
                                               (1e9, W.MAT_WATER, 1.0)])
    return W.homogeneous(dims, case["voxel"], W.MAT_WATER, 1.0)


def _resident(ctx, case, dims, seed):
    if case["phantom"] == "noise":
        mat, rho = _density_field(*dims, case["voxel"], seed)
        torch.cuda.synchronize()
        return ctx.create_phantom_device(dims, (case["voxel"],) * 3, mat.data_ptr(), rho.data_ptr())
    return ctx.create_phantom(_phantom(case, dims, seed))


def _source(case, particle, dims, energy, field, seed):
    X, Y = dims[0] * case["voxel"], dims[1] * case["voxel"]
    kind = W.ELECTRON if particle == "electron" else W.PHOTON
    center = (X / 2, Y / 2)
    if case["source"] == "phsp":
        ph = W.Phantom(dims, (case["voxel"],) * 3, np.empty(0), np.empty(0))
        n = max(1000, min(case["histories"], 200_000))
        rng = np.random.default_rng(seed)
        e = W.draw_spectrum(*W.synthetic_6mv_spectrum(), n, seed) if kind == W.PHOTON else 1.0 + 14.0 * rng.random(n)
        src = W.point_source_phase_space(kind, ph, n, seed, field_cm=field, energies=e)
        src.energy_grouping = W.ENERGY_GROUPED
        return src
    if case["source"] in ("spectrum", "grouped"):
        edges, w = (W.synthetic_6mv_spectrum() if kind == W.PHOTON
                    else (np.linspace(1.0, 15.0, 15), np.full(14, 1.0 / 14)))
        return W.Source(kind, W.BEAM_SQUARE, center_cm=center, field_cm=field, spectrum_edges=edges,
                        spectrum_weights=w, energy_grouping=W.ENERGY_GROUPED if case["source"] == "grouped"
                        else W.ENERGY_UNGROUPED)
    if field == 0.0:
        return W.pencil(kind, energy, *center)
    return W.Source(kind, W.BEAM_SQUARE, energy=energy, center_cm=center, field_cm=field)


class _State:
    """A program's handles and buffers; phantoms and plans go when it goes."""

    def __init__(self, case, ctx):
        self.case, self.ctx = case, ctx
        self.phantoms, self.plans, self.sources, self.seeds, self.histories, self.out = [], [], [], [], [], []

    def __del__(self):
        try:
            for p in self.plans:
                self.ctx.plan_close(p)
            for p in self.phantoms:
                self.ctx.destroy_phantom(p)
        except Exception:
            pass


def _uneven(case):
    """The plans of a many-plan case: sizes, energies, fields and counts spread about the case's own.
    They are the case's, not the seed's, so that another seed is the same work."""
    r = random.Random(case["nx"] * 1000003 + case["ny"] * 1009 + case["nz"])
    for i in range(case["plans"]):
        lo, hi = sorted((case["nx"], case["nz"]))
        n = r.randint(lo, hi) if hi > lo else lo
        yield ((n, max(lo, n - r.randint(0, 9)), n), "electron" if i % 2 == 0 else "photon",
               round(case["energy"] * r.uniform(0.5, 1.0), 2), round(case["field"] * r.uniform(0.4, 1.0), 2),
               max(1, int(case["histories"] * _log(r, 0.1, 1.0))))


def prepare(case, seed):
    ctx = _engine(case)
    s = _State(case, ctx)
    dims = (case["nx"], case["ny"], case["nz"])
    if case["form"] in ("batch", "target", "served"):
        todo = list(_uneven(case))
    else:
        todo = [(dims, case["particle"], case["energy"], case["field"], case["histories"])]
    for i, (d, particle, energy, field, n) in enumerate(todo):
        own = seed * 64 + i + 1
        src = _source(case, particle, d, energy, field, own)
        s.sources.append(src)
        s.seeds.append(own * 0x9E3779B97F4A7C15 % (1 << 62))
        s.histories.append(n)
        nvox = d[0] * d[1] * d[2]
        if case["form"] == "e2e":
            s.host = (_phantom(case, d, own) if case["phantom"] != "noise" else _from_device(case, d, own))
        else:
            s.phantoms.append(_resident(ctx, case, d, own))
        if case["form"] in ("simulate", "e2e"):
            s.out = [torch.empty(nvox, dtype=torch.float64, pin_memory=True).numpy() for _ in range(2)]
        elif case["form"] != "served":
            s.plans.append(ctx.plan_open(s.phantoms[-1], src, s.seeds[-1], case["batches"]))
            s.out.append([torch.empty(nvox, dtype=torch.float64, device="cuda") for _ in range(2)])
        else:
            s.out.append(nvox)
    if case["form"] == "readout":
        ctx.run(s.plans, s.histories)
    return s


def _from_device(case, dims, seed):
    mat, rho = _density_field(*dims, case["voxel"], seed)
    return W.Phantom(dims, (case["voxel"],) * 3, mat.cpu().numpy(), rho.cpu().numpy())


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _numbers(stats):
    return np.array([stats[k] for k in COUNTS], dtype=np.int64), np.array([stats["d_max_gy"], stats["s_thr"]])


def _results(s):
    out = []
    for plan, (dose, sigma) in zip(s.plans, s.out):
        st = s.ctx.plan_result(plan, 0.5, dose.data_ptr(), sigma.data_ptr())
        out.append([dose, sigma, *_numbers(st)])
    return out


def run(state):
    s, ctx, form = state, state.ctx, state.case["form"]
    if form == "simulate":
        r = ctx.simulate(s.phantoms[0], s.sources[0], s.histories[0], s.seeds[0], out=s.out)
        return [r.dose, r.sigma, *_numbers(r.stats)]
    if form == "e2e":
        pid = ctx.create_phantom(s.host)
        r = ctx.simulate(pid, s.sources[0], s.histories[0], s.seeds[0], out=s.out)
        ctx.destroy_phantom(pid)
        return [r.dose, r.sigma, *_numbers(r.stats)]
    if form == "served":
        srv = serve.Server(ctx, 64 << 30, target=s.case["target"], n_batches=s.case["batches"],
                           first_chunk=s.case["histories"], keep_dose=True)
        for i, (pid, src, seed, nvox) in enumerate(zip(s.phantoms, s.sources, s.seeds, s.out)):
            srv.submit(serve.DoseRequest(i, pid, nvox, src, seed, max_histories=20_000_000))
        done = sorted(srv.run(real_time=False), key=lambda r: r.rid)
        return [[r.dose, r.sigma, r.histories, r.s_thr] for r in done]
    if form == "readout":
        return _results(s)
    for plan, seed in zip(s.plans, s.seeds):
        ctx.plan_reset(plan, seed)
    if form == "target":
        got = ctx.run_to_uncertainty(s.plans, s.histories, [20_000_000] * len(s.plans), s.case["target"])
        return [_results(s), np.array(got["histories"], dtype=np.int64), np.array(got["s_thr"]), got["rounds"]]
    ctx.run(s.plans, s.histories)
    return _results(s)


# ---------------------------------------------------------------------------
# The least work of a pass
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: each phantom's words read (host arrays uploaded), each batch tally zeroed and folded, dose and
    sigma written.  Operations: about 500 for each electron step and photon flight, of which a history takes
    about 5 for each MeV of an electron beam and 3 for each MeV of a photon beam that is absorbed."""
    if case["form"] in ("batch", "target", "served"):
        todo = list(_uneven(case))
    else:
        todo = [((case["nx"], case["ny"], case["nz"]), case["particle"], case["energy"], case["field"],
                 case["histories"])]
    size = ops = 0.0
    for d, particle, energy, field, n in todo:
        nvox = d[0] * d[1] * d[2]
        mev = energy if case["source"] == "mono" else 8.0 if particle == "electron" else 1.5
        if case["target"]:  # a voxel of the high-dose region needs about 1/target^2 crossings
            cross = (field / case["voxel"]) ** 2 / case["target"] ** 2
            n = max(n, min(2e7, cross * (0.5 if particle == "electron" else 10.0)))
        tallies = 8.0 * case["batches"] * nvox
        size += (5.0 if case["form"] == "e2e" else 4.0) * nvox + 16.0 * nvox + tallies
        if case["form"] != "readout":
            size += tallies
            steps = 3.0 if case["kerma"] else mev * (5.0 if particle == "electron" else 3.0)
            ops += 500.0 * n * steps
    return {"bytes": size, "flops": ops}


def exact(case, seed):
    """No other program gives a keyed Monte Carlo's own histories, in 64 bits or any other."""
    return None
