"""Workloads on which the transport library's speed is measured, through its Python API.

Each case is one whole use of the library as a program makes it: reset the tally, inject a
pool, advance it (or run the adjoint, or convert a background), and hand back the particles,
the tally with its batch-means classes and the ledger.  The background, the pool's and the
tally's memory and the scratch workspace are prepared once, as a program keeps them.

Kinds
  advance   one parameter set on a uniform or radially stretched grid
  amr       one parameter set on a block-AMR grid
  ensemble  many parameter sets in one pool
  stream    snapshots streamed from page-locked host memory through a ring of device slots
  adjoint   forward and reverse pass of a smooth observable
  convert   FP32 background to 16-bit and / or pair records

Winds, injections, observers and sizes are those of fte_inputs.configs, the tests and the
benchmark; the seed sets the random streams of the particles and the speeds and field
strength of the wind.
"""
import dataclasses
import functools
import math
import random

import numpy as np
import torch

from fte_inputs import amr, backgrounds, configs
from fte_inputs.configs import InjectSpec, Observer, Params, SmoothObserver
from fte_inputs.grid import REC, GridSpec
from paper_2404_12164_gb300 import api

DEG = math.pi / 180.0
F64 = torch.float64

# Defaults of a case; a listed or drawn case states what differs from them.
DEFAULTS = dict(wind="cir", nr=512, nth=60, nph=180, radial="linear", snaps=24, periodic=True,
                store="f32", layout="cell", model="qlt", lam=0.1, perp=0.0, energy="mono", e0=0.05,
                dt=10.0, sort=64, tally="global", obs="box", nt=144, p_update="exp")


def _case(kind, name=None, **kw):
    c = {"kind": kind, **DEFAULTS, **kw}
    return {"name": name, **c} if name else c


def listed():
    return [
        # A first look or a unit check: a small pool for a few hundred steps, where launches and
        # the latency of one step decide (the smoke run's size).
        _case("advance", "parker_short", wind="parker", nr=128, nth=16, nph=32, snaps=1, n=2000, steps=200,
              lam=0.3, e0=0.1, sort=0, obs="near"),
        # The Parker workload as configured: 1e4 protons for one day, one launch after another of
        # a pool that fills an eighth of the GPU's threads.
        _case("advance", "parker_day", wind="parker", nr=128, nth=16, nph=32, snaps=1, n=10_000, steps=8640,
              lam=0.3, e0=0.1, sort=0, obs="shell"),
        # The headline run: 1e6 protons over 4 days of 24 hourly snapshots (12.7 GB).
        _case("advance", "cir_4days", n=1_000_000, steps=34_560),
        # The same wind stored in BF16, a quarter of a day with a pool of ordinary size.
        _case("advance", "cir_bf16_6h", store="bf16", n=300_000, steps=2160),
        # Cross-field diffusion with Eq. 5's pitch-angle coefficient, a power-law spectrum and
        # all four observer kinds: the physics options a study of profiles switches on.
        _case("advance", "cir_perp_profiles", nr=256, nth=30, nph=90, snaps=3, periodic=False, n=120_000,
              steps=96, model="paper", perp=3e-4, energy="powerlaw", obs="all", nt=72),
        # A radially stretched grid of odd sizes in FP16 pair records, isotropic scattering,
        # shared-memory tally and a ragged pool that is not reordered.
        _case("advance", "log_f16_odd", nr=97, nth=31, nph=53, radial="log", snaps=5, store="f16", layout="pair",
              n=33_333, steps=300, model="iso", p_update="euler", sort=0, tally="shared", obs="slab", nt=36),
        # The block-AMR workload with its two coarser levels (11,296 leaves, 12.7 GB) and its pool
        # of 1e7 protons, for the first ten simulated minutes.
        _case("amr", "amr_band", nr=32, nth=8, nph=24, bsize=16, levels=2, snaps=2, periodic=False, radial="log",
              threshold=6e-5, n=10_000_000, steps=320, dt=2.0, energy="powerlaw", obs="band"),
        # A parameter study: 64 sets of unequal size over 1.5 hours.
        _case("ensemble", "ensemble_64", nr=256, nth=30, nph=90, sets=64, n=4_000_000, steps=540),
        # A day with 24 snapshots streamed through four device slots, as where the sequence does
        # not fit the device.
        _case("stream", "stream_day", nr=256, nth=30, nph=90, ring=4, n=300_000, steps=8640),
        # One gradient evaluation of a fit, through torch.autograd, at a fifth of the headline pool.
        _case("adjoint", "fit_gradient", snaps=4, periodic=False, n=200_000, steps=1024, every=256,
              energy="powerlaw", autograd=True),
        # Per-particle gradients on a small pool (a test or a sensitivity map), Eq. 5's model,
        # not reordered.
        _case("adjoint", "sensitivity_map", nr=128, nth=30, nph=90, snaps=3, periodic=False, n=20_000, steps=400,
              every=64, model="paper", energy="powerlaw", sort=0, autograd=False),
        # Loading a sequence in BF16: 24 FP32 snapshots converted on the device.
        _case("convert", "convert_bf16", store="bf16"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 5 + ["amr", "ensemble", "stream", "adjoint", "adjoint", "convert"])
    grid = dict(nr=_logint(rng, 65, 512), nth=rng.randint(15, 60), nph=rng.randint(31, 180),
                radial=rng.choice(["linear", "linear", "log"]), snaps=rng.randint(2, 24))
    grid["periodic"] = grid["snaps"] > 6
    phys = dict(model=rng.choice(["qlt", "qlt", "paper", "iso"]), energy=rng.choice(["mono", "powerlaw"]),
                lam=round(rng.uniform(0.05, 1.0), 3))
    store = dict(store=rng.choice(["f32", "f32", "bf16", "f16"]), layout=rng.choice(["cell", "cell", "cell", "pair"]))
    if kind == "advance":
        n = _logint(rng, 1000, 1_000_000)
        steps = _logint(rng, 50, min(34_560, 10_000_000_000 // n))
        shared = rng.random() < 0.15
        return _case(kind, **grid, **phys, **store, n=n, steps=steps, perp=rng.choice([0.0, 0.0, 0.0, 3e-4]),
                     sort=0 if n < 20_000 else rng.choice([0, 32, 64, 64]), tally="shared" if shared else "global",
                     obs=rng.choice(["box", "shell", "slab"]), nt=36 if shared else 144,
                     p_update=rng.choice(["exp", "exp", "euler"]))
    if kind == "amr":
        n = _logint(rng, 30_000, 10_000_000)
        return _case(kind, nr=8, nth=4, nph=8, bsize=rng.choice([8, 16]), levels=rng.choice([2, 3]), radial="log",
                     snaps=2, periodic=False, threshold=1e-5, n=n, steps=_logint(rng, 64, 640), dt=2.0, obs="band",
                     store=store["store"], energy="powerlaw")
    if kind == "ensemble":
        return _case(kind, **grid, **store, sets=rng.randint(2, 64), n=_logint(rng, 60_000, 4_000_000),
                     steps=_logint(rng, 64, 540), model=phys["model"])
    if kind == "stream":
        snaps = rng.randint(7, 24)
        return _case(kind, nr=_logint(rng, 65, 256), nth=rng.randint(15, 30), nph=rng.randint(31, 90), snaps=snaps,
                     ring=rng.randint(3, min(snaps, 6)), n=_logint(rng, 20_000, 300_000), steps=_logint(rng, 400, 8640),
                     store=rng.choice(["f32", "f32", "bf16"]))
    if kind == "adjoint":
        n = _logint(rng, 2000, 200_000)
        return _case(kind, **grid, **phys, store=store["store"], layout=store["layout"], n=n,
                     steps=_logint(rng, 100, 1024), every=rng.choice([64, 100, 256]),
                     sort=0 if n < 20_000 else rng.choice([32, 64]), autograd=rng.random() < 0.5)
    if store["store"] == "f32":
        store["layout"] = "pair"
    return _case(kind, **grid, **store)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _wind(case, seed):
    """Keyword arguments of the analytic wind: speeds and field strength set by the seed."""
    r = random.Random(seed)
    if case["wind"] == "parker":
        return dict(v_kms=r.uniform(380.0, 420.0), b1_nt=r.uniform(4.5, 5.5))
    return dict(v_slow=r.uniform(320.0, 340.0), v_fast=r.uniform(680.0, 720.0), br_b=r.uniform(330.0, 370.0))


def _grid(case):
    return GridSpec(nr=case["nr"], nth=case["nth"], nph=case["nph"], radial=case["radial"], n_snap=case["snaps"],
                    periodic=case["periodic"], t_snap0=0.0, dt_snap=3600.0)


def _centres(g, device):
    i = torch.arange(g.nr, dtype=F64, device=device) + 0.5
    if g.radial == "log":
        r = g.r_min * torch.exp(i * (math.log(g.r_max / g.r_min) / g.nr))
    else:
        r = g.r_min + i * ((g.r_max - g.r_min) / g.nr)
    th = g.th_min + (torch.arange(g.nth, dtype=F64, device=device) + 0.5) * ((g.th_max - g.th_min) / g.nth)
    ph = (torch.arange(g.nph, dtype=F64, device=device) + 0.5) * (2.0 * math.pi / g.nph)
    return r, th, ph


def _fill_fields(case, g, out, wind):
    """Cell records [snap][phi][theta][r][24] of the analytic wind with gridded gradients (what a
    post-processor of MHD output delivers), evaluated on out's device."""
    r, th, ph = _centres(g, out.device)
    R, TH, PH = r[None, None, :], th[None, :, None], ph[:, None, None]
    shape = (g.nph, g.nth, g.nr)
    st, ct, sp, cp = torch.sin(TH), torch.cos(TH), torch.sin(PH), torch.cos(PH)
    rhat = (st * cp, st * sp, ct)
    that = (ct * cp, ct * sp, -st)
    phat = (-sp, cp, torch.zeros_like(sp))
    dph = 2.0 * math.pi / g.nph

    def grad(f):
        fr, ft = torch.gradient(f, spacing=(r, th), dim=(2, 1), edge_order=2)
        fp = (torch.roll(f, -1, 0) - torch.roll(f, 1, 0)) / (2.0 * dph)
        ft, fp = ft / R, fp / (R * st)
        return [fr * rhat[j] + ft * that[j] + fp * phat[j] for j in range(3)]

    out[..., 18:] = 0.0
    for s in range(g.n_snap):
        if case["wind"] == "parker":
            B, V = backgrounds.parker_fields(R, TH, PH, **wind)
        else:
            B, V = backgrounds.cir_fields(R, TH, PH, g.t_snap0 + s * g.dt_snap, **wind)
        B = [b.expand(shape) for b in B]
        V = [v.expand(shape) for v in V]
        o = out[s]
        for i in range(3):
            o[..., i] = B[i]
            o[..., 3 + i] = V[i]
            for j, d in enumerate(grad(V[i])):
                o[..., 6 + 3 * i + j] = d
        for j, d in enumerate(grad(torch.sqrt(B[0] ** 2 + B[1] ** 2 + B[2] ** 2))):
            o[..., 15 + j] = d


def _inject(case, seed):
    key = dict(seed=seed & 0xFFFFFFFF)
    if case["energy"] == "mono":
        key.update(energy="mono", e0=case["e0"])
    else:
        key.update(energy="powerlaw", e1=0.05, e2=5.0, gamma=3.0)
    if case["wind"] == "parker":
        return InjectSpec(region="point", r=0.1, th=90 * DEG, ph=0.0, weight="unit", **key)
    if case["kind"] == "amr":
        return dataclasses.replace(configs.cir_amr_1e7(spec=_amr_spec(case)).inject, **key)
    return InjectSpec(region="box", r1=1.0, r2=2.0, th1=88 * DEG, th2=92 * DEG, ph1=math.pi, ph2=2 * math.pi,
                      divv_max=0.0, divv_snap=0, weight="r-2", **key)


def _params(case, seed):
    return Params(dmumu=case["model"], lambda_par=case["lam"], lambda_perp=case["perp"], dt=case["dt"],
                  p_update=case["p_update"], seed=seed & 0xFFFFFFFF, sort_every=case["sort"],
                  tally_layout=case["tally"])


def _observers(case):
    t_end = max(case["steps"] * case["dt"], 1.0)
    common = dict(ne=16, t_lo=0.0, t_hi=t_end, nt=case["nt"])
    box = dict(kind="box", dr=0.02, th=90 * DEG, dth=2 * DEG, dph=2 * DEG, e_lo=0.01, e_hi=10.0, **common)
    if case["obs"] == "shell":
        return [Observer(kind="shell", r=1.0, dr=0.01, e_lo=0.01, e_hi=1.0, **common)]
    if case["obs"] == "near":              # a shell that protons from 0.1 au reach within minutes
        return [Observer(kind="shell", r=0.12, dr=0.01, e_lo=0.01, e_hi=1.0, **common)]
    if case["obs"] == "slab":              # x = -1 au cuts the injected CIR
        return [Observer(kind="slab", r=-1.0, dr=0.05, e_lo=0.01, e_hi=10.0, **common)]
    if case["obs"] == "band":
        return [Observer(r=r, ph=configs.cir_observer_phi(r), **box) for r in (0.5, 1.0, 1.5, 1.8)]
    if case["obs"] == "all":
        return [Observer(r=1.0, ph=configs.cir_observer_phi(1.0), **box),
                Observer(kind="shell", r=1.2, dr=0.01, e_lo=0.01, e_hi=10.0, **common),
                Observer(kind="slab", r=-1.0, dr=0.05, e_lo=0.01, e_hi=10.0, **common),
                Observer(kind="ring", r=1.5, dr=0.05, th=90 * DEG, dth=2 * DEG, e_lo=0.01, e_hi=10.0, **common)]
    return [Observer(r=1.0, ph=configs.cir_observer_phi(1.0), **box)]


def _smooth(case):
    t_end = case["steps"] * case["dt"]
    return SmoothObserver(r_o=1.15, sigma_r=0.05, e_c=0.08, sigma_lnE=0.5, t_c=0.75 * t_end, sigma_t=0.5 * t_end)


def _cell_background(case, seed):
    g = _grid(case)
    bg = api.Background(g)
    _fill_fields(case, g, bg.dev.view(g.n_snap, g.nph, g.nth, g.nr, REC), _wind(case, seed))
    return bg


def _stored(case, cell):
    """The background in the case's storage form."""
    if case["store"] == "f32" and case["layout"] == "cell":
        return cell
    if case["kind"] == "amr":
        bg = api.AmrBackground(cell.grid, cell.leaves, dtype=case["store"], layout=case["layout"], share=cell)
    else:
        bg = api.Background(cell.grid, dtype=case["store"], layout=case["layout"])
    api.fte_quantize_background(bg, cell)
    return bg


def _amr_spec(case):
    return amr.AmrSpec(nbr=case["nr"], nbt=case["nth"], nbp=case["nph"], bsize=case["bsize"], levels=case["levels"],
                       radial=case["radial"], n_snap=case["snaps"], periodic=case["periodic"], t_snap0=0.0,
                       dt_snap=3600.0)


@functools.lru_cache(maxsize=4)
def _amr_leaves(nbr, nbt, nbp, bsize, levels, radial, threshold):
    spec = amr.AmrSpec(nbr=nbr, nbt=nbt, nbp=nbp, bsize=bsize, levels=levels, radial=radial, n_snap=2,
                       periodic=False, t_snap0=0.0, dt_snap=3600.0)
    return amr.build_leaves(spec, amr.divv_refiner_batched(spec, threshold, device="cuda"))


def _amr_background(case, seed):
    spec = _amr_spec(case)
    leaves = _amr_leaves(case["nr"], case["nth"], case["nph"], case["bsize"], case["levels"], case["radial"],
                         case["threshold"])
    bg = api.AmrBackground(spec, leaves)
    bg.leaves = leaves
    P = spec.bsize + 2
    view = bg.dev.view(spec.n_snap, len(leaves), P, P, P, REC)
    view.zero_()
    amr.fields_batched(spec, leaves, device="cuda", out=view, **_wind(case, seed))
    api.fte_amr_prepare(bg)
    return bg


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind == "convert":
        s.src = _cell_background(case, seed)
        s.bg = api.Background(s.src.grid, dtype=case["store"], layout=case["layout"])
        return s
    s.inject, s.params = _inject(case, seed), _params(case, seed)
    if kind == "stream":
        g = _grid(case)
        dev = torch.empty((g.n_snap, g.nph, g.nth, g.nr, REC), dtype=torch.float32, device="cuda")
        _fill_fields(case, g, dev, _wind(case, seed))
        host = torch.empty(dev.shape, dtype=torch.float32, pin_memory=True)
        host.copy_(dev)
        del dev
        s.bg = api.Background(g, dtype=case["store"], ring=case["ring"])
        s.snaps = api.SnapshotStream(s.bg, host)
    elif kind == "amr":
        s.bg = _stored(case, _amr_background(case, seed))
    else:
        s.bg = _stored(case, _cell_background(case, seed))
    if kind == "adjoint":
        s.obs = _smooth(case)
        if case["autograd"]:        # `run` of api.SmoothIntensity
            s.run = _State()
            s.run.bg, s.run.params, s.run.inject, s.run.obs = s.bg, s.params, s.inject, s.obs
            s.run.n_steps, s.run.n_particles, s.run.checkpoint_every = case["steps"], case["n"], case["every"]
            return s
        s.tally = api.Tally([])
        s.pool = api.Particles(case["n"])
        s.adj = api.Adjoint(s.bg, s.params, s.obs, 0, case["steps"], case["every"], ws=api.Workspace())
        return s
    s.pool = api.Particles(case["n"])
    s.ws = api.Workspace()
    if kind == "ensemble":
        s.sets = configs.ensemble_sets(case["sets"], case["n"], base_inject=s.inject, rng_seed=seed)
        s.tally = api.Tally(_observers(case), n_sets=case["sets"])
    else:
        s.tally = api.Tally(_observers(case))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _pool_out(pool):
    n = pool.count
    return {k: getattr(pool, k)[:n] for k in ("x", "y", "z", "mu", "p", "w", "id", "status")}


def _tally_out(t):
    return {"S": t.S, "S2": t.S2, "C": t.C, "S_class": t.S_class, "ledger_w": t.ledger_w, "ledger_n": t.ledger_n}


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "convert":
        api.fte_quantize_background(s.bg, s.src)
        return {"records": s.bg.dev.view(torch.uint8)[: s.bg.nbytes]}
    if kind == "adjoint" and case["autograd"]:
        p = s.params
        theta = torch.tensor([p.lambda_par, p.q, p.H, p.eps, s.inject.gamma], dtype=F64, requires_grad=True)
        J = api.SmoothIntensity.apply(theta, s.run)
        J.backward()
        return {"J": J.detach(), "grad": theta.grad}
    s.pool.c.count = 0
    api.fte_tally_reset(s.tally)
    if kind == "ensemble":
        api.fte_inject_batched(s.pool, s.bg, s.sets, s.tally)
        api.fte_advance_batched(s.pool, s.bg, s.params, s.sets, s.tally, 0, case["steps"], s.ws)
        return {**_pool_out(s.pool), **_tally_out(s.tally)}
    if kind == "stream":
        s.snaps.slots[:] = -1              # a new sequence: nothing of it is on the device yet
        s.snaps.load(0)
        api.fte_inject(s.pool, s.bg, s.inject, case["n"], s.tally, check_failed=False)
        api.fte_advance_streamed(s.pool, s.bg, s.snaps, s.params, s.tally, 0, case["steps"], s.ws)
        return {**_pool_out(s.pool), **_tally_out(s.tally)}
    api.fte_inject(s.pool, s.bg, s.inject, case["n"], s.tally, id_base=0, check_failed=False)
    if kind == "adjoint":
        J, Ji = s.adj.forward(s.pool, per_particle=True)
        grad, pp = s.adj.reverse(s.pool, s.inject, per_particle=True)
        return {"J": J, "J_i": Ji, "grad": grad, "per_particle": pp, **_pool_out(s.pool)}
    api.fte_advance(s.pool, s.bg, s.params, s.tally, 0, case["steps"], s.ws)
    return {**_pool_out(s.pool), **_tally_out(s.tally)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# floating operations of one particle-step: 16 records x 18 fields of multiply-add, and about
# 350 for locating, the coefficients, one Philox block's normals and the update; the reverse
# pass re-evaluates the step and runs its vector-Jacobian product (about 2.2 forward steps)
STEP_FLOPS = 16 * 18 * 2 + 350
PERP_FLOPS = 16 * 9 * 2 + 120
REC_BYTES = {"f32": 72, "bf16": 36, "f16": 36}


def _alive_steps(case):
    """Particle-steps of a run.  Protons of the CIR injection leave the domain over about 1.3e5 s;
    the other runs are short against that or stay inside."""
    tau = 1.3e5 if case["wind"] == "cir" and case["kind"] != "amr" else 1e9
    t = case["steps"] * case["dt"]
    return case["n"] * case["steps"] * (tau / t) * -math.expm1(-t / tau)


def work(case):
    cells = case["nr"] * case["nth"] * case["nph"]
    rec = REC_BYTES[case["store"]]
    if case["kind"] == "convert":
        pair = case["layout"] == "pair"
        out = (160 if pair else 96) if case["store"] == "f32" else (96 if pair else 64)
        return {"bytes": cells * case["snaps"] * (72 + out), "flops": cells * case["snaps"] * 18 * 2}
    if case["kind"] == "amr":
        cells *= case["bsize"] ** 3
    steps = _alive_steps(case)
    used = min(case["snaps"], 2 + int(case["steps"] * case["dt"] / 3600.0)) if case["snaps"] > 1 else 1
    # the records that the pool visits: at most the stored ones, at most 16 a particle-step
    field_bytes = min(cells * used * rec, 16 * rec * steps)
    if case["kind"] == "stream":
        field_bytes = cells * used * 96
    pool = 2 * 25 * case["n"]
    flops = steps * (STEP_FLOPS + (PERP_FLOPS if case["perp"] > 0 else 0))
    if case["kind"] == "adjoint":
        flops *= 4.2
        pool += 2 * 20 * case["n"] * -(-case["steps"] // case["every"])
    return {"bytes": field_bytes + pool, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
C_AU = 2.003988804e-3            # speed of light, au/s
MC2 = 938.27208816               # proton rest energy, MeV
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    c = [torch.as_tensor(v, dtype=torch.int64, device=c1.device).expand_as(c1) for v in (c0, c1, c2, c3)]
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & M32) ^ c[1] ^ k0, b & M32, ((a >> 32) & M32) ^ c[3] ^ k1, a & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _u(x):
    return ((x >> 8).to(F64) + 0.5) / 16777216.0


def _exact_fields(case, seed):
    """The stored values of the background as 64-bit numbers [snap * cells, 18]."""
    g = _grid(case)
    f = torch.empty((g.n_snap, g.nph, g.nth, g.nr, REC), dtype=torch.float32, device="cuda")
    _fill_fields(case, g, f, _wind(case, seed))
    f = f.view(-1, REC)[:, :18]
    if case["store"] == "f32":
        return f.to(F64)
    sc = f.abs().amax(dim=0)
    sc = torch.where(sc > 0, sc, torch.ones_like(sc))
    h = (f / sc).to(torch.bfloat16 if case["store"] == "bf16" else torch.float16)
    return h.to(F64) * sc.to(F64)


def _exact_inject(case, seed, fields):
    sp, g, n = _inject(case, seed), _grid(case), case["n"]
    pid = torch.arange(n, dtype=torch.int64, device="cuda")
    d = _philox(0, pid, 1, 0, sp.seed, sp.set_id)
    mu = 2.0 * _u(d[0]) - 1.0
    if sp.energy == "mono":
        E = torch.full_like(mu, sp.e0)
    else:
        g1 = 1.0 - sp.gamma
        E = (sp.e1 ** g1 + _u(d[1]) * (sp.e2 ** g1 - sp.e1 ** g1)) ** (1.0 / g1)
    T = E / MC2
    p = torch.sqrt(T * (T + 2.0))
    r, th, ph = torch.full_like(mu, sp.r), torch.full_like(mu, sp.th), torch.full_like(mu, sp.ph)
    if sp.region == "box":
        todo = pid
        f32 = fields.float()
        for t in range(sp.max_tries):
            q = _philox(t, todo, 2, 0, sp.seed, sp.set_id)
            rr = (sp.r1 ** 3 + _u(q[0]) * (sp.r2 ** 3 - sp.r1 ** 3)) ** (1.0 / 3.0)
            tt = torch.acos(math.cos(sp.th1) + _u(q[1]) * (math.cos(sp.th2) - math.cos(sp.th1)))
            pp = sp.ph1 + _u(q[2]) * (sp.ph2 - sp.ph1)
            r[todo], th[todo], ph[todo] = rr, tt, pp
            xr = torch.log(rr / g.r_min) / math.log(g.r_max / g.r_min) if g.radial == "log" else \
                (rr - g.r_min) / (g.r_max - g.r_min)
            ci = (xr * g.nr).floor().long().clamp(0, g.nr - 1)
            cj = ((tt - g.th_min) / (g.th_max - g.th_min) * g.nth).floor().long().clamp(0, g.nth - 1)
            ck = (torch.remainder(pp, 2 * math.pi) / (2 * math.pi) * g.nph).floor().long() % g.nph
            rec = f32[(sp.divv_snap * g.nph + ck) * g.nth * g.nr + cj * g.nr + ci]
            ok = rec[:, 6] + rec[:, 10] + rec[:, 14] < sp.divv_max
            todo = todo[~ok]
            if todo.numel() == 0:
                break
    w = 1.0 / r ** 2 if sp.weight == "r-2" else torch.ones_like(r)
    st = torch.sin(th)
    return dict(x=r * st * torch.cos(ph), y=r * st * torch.sin(ph), z=r * torch.cos(th), mu=mu, p=p, w=w), pid


def _norm(prm):
    """Integral that ties D_mumu to lambda_par (Simpson in s, mu = s^3)."""
    m = np.linspace(0.0, 1.0, 16385)
    u, m = m, m ** 3
    if prm.dmumu == "qlt":
        den = m ** (prm.q - 1.0) + prm.H
    else:
        den = m / (1.0 + m) + prm.eps
    f = 3.0 * u * u * (1.0 - m * m) / den
    wgt = np.ones_like(u)
    wgt[1:-1:2], wgt[2:-1:2] = 4.0, 2.0
    return float((wgt * f).sum() / (3.0 * 16384))


def _snap_pair(g, t):
    if g.n_snap == 1:
        return 0, 0, 0.0, False
    tau = (t - g.t_snap0) / g.dt_snap
    k = math.floor(tau)
    if g.periodic:
        return k % g.n_snap, (k + 1) % g.n_snap, tau - k, True
    if tau < 0 or tau >= g.n_snap - 1:
        s = 0 if tau < 0 else g.n_snap - 1
        return s, s, 0.0, False
    return k, k + 1, tau - k, True


def _axis(x, n):
    """Lower cell, weight and derivative flag on an axis that is held constant past its centres."""
    lo, hi = x < 0, x >= n - 1
    i = torch.where(hi, torch.full_like(x, n - 2), torch.where(lo, torch.zeros_like(x), x.floor())).long()
    w = torch.where(hi, torch.ones_like(x), torch.where(lo, torch.zeros_like(x), x - i))
    return i, w, (~(lo | hi)).to(F64)


def _exact_step(case, g, prm, I, fields, n, pid, q):
    """One Euler-Maruyama step of the focused transport equation; returns the new state and the
    start-of-step (r, theta, phi)."""
    x, y, z, mu, p = q["x"], q["y"], q["z"], q["mu"], q["p"]
    rho = torch.sqrt(x * x + y * y)
    r = torch.sqrt(x * x + y * y + z * z)
    th, ph = torch.atan2(rho, z), torch.remainder(torch.atan2(y, x), 2 * math.pi)
    s0, s1, wt, two = _snap_pair(g, prm.t0 + n * prm.dt)
    if g.radial == "log":
        dl = math.log(g.r_max / g.r_min) / g.nr
        i, _, on = _axis(torch.log(r / g.r_min) / dl - 0.5, g.nr)
        c0, c1 = g.r_min * torch.exp((i + 0.5) * dl), g.r_min * torch.exp((i + 1.5) * dl)
        fr = torch.where(on > 0, (r - c0) / (c1 - c0), (i > 0).to(F64))
        dfr = on / (c1 - c0)
    else:
        dr = (g.r_max - g.r_min) / g.nr
        i, fr, on = _axis((r - g.r_min) / dr - 0.5, g.nr)
        dfr = on / dr
    dth = (g.th_max - g.th_min) / g.nth
    j, ft, on = _axis((th - g.th_min) / dth - 0.5, g.nth)
    dft = on / dth
    dph = 2 * math.pi / g.nph
    xk = ph / dph - 0.5
    k = xk.floor()
    fp = xk - k
    k = k.long() % g.nph
    cells = g.nr * g.nth * g.nph
    F = torch.zeros((x.numel(), 18), dtype=F64, device=x.device)
    dv = torch.zeros((x.numel(), 3), dtype=F64, device=x.device)
    dB = [torch.zeros_like(dv) for _ in range(3)]
    for snap, ws, sgn in ((s0, 1.0 - wt, -1.0), (s1, wt, 1.0)) if two else ((s0, 1.0, 0.0),):
        for c in range(8):
            a, b, e = c & 1, (c >> 1) & 1, c >> 2
            wr, wth, wph = (fr if a else 1 - fr), (ft if b else 1 - ft), (fp if e else 1 - fp)
            f = fields[snap * cells + (((k + e) % g.nph) * g.nth + j + b) * g.nr + i + a]
            w8 = (wr * wth * wph)[:, None]
            F += ws * w8 * f
            dv += sgn * w8 * f[:, 3:6]
            if prm.lambda_perp > 0:
                B3 = ws * f[:, :3]
                dB[0] += ((1 if a else -1) * dfr * wth * wph)[:, None] * B3
                dB[1] += ((1 if b else -1) * dft * wr * wph)[:, None] * B3
                dB[2] += ((1 if e else -1) / dph * wr * wth)[:, None] * B3
    B, V, G, gB = F[:, 0:3], F[:, 3:6], F[:, 6:15].view(-1, 3, 3), F[:, 15:18]
    Bm = B.norm(dim=1)
    b = B / Bm[:, None]
    divb = -(b * gB).sum(1) / Bm
    divv = G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2]
    bbgv = torch.einsum("ni,nij,nj->n", b, G, b)
    bdvdt = torch.zeros_like(x)
    if prm.dvdt_term:
        acc = torch.einsum("nij,nj->ni", G, V) + (dv / g.dt_snap if two else 0.0)
        bdvdt = (b * acc).sum(1)
    v = C_AU * p / torch.sqrt(1 + p * p)
    am, sg, omm = mu.abs(), torch.sign(mu), 1 - mu * mu
    if prm.dmumu == "qlt":
        nu = 1.5 * v * I / prm.lambda_par
        h = am ** (prm.q - 1) + prm.H
        dh = (prm.q - 1) * am.clamp(min=prm.mu_floor) ** (prm.q - 2) * sg
        D, dD = 0.5 * nu * omm * h, 0.5 * nu * (omm * dh - 2 * mu * h)
    elif prm.dmumu == "paper":
        D0 = 0.75 * v * I / prm.lambda_par
        h, dh = am / (1 + am) + prm.eps, sg / (1 + am) ** 2
        D, dD = D0 * h * omm, D0 * (dh * omm - 2 * mu * h)
    else:
        D = 0.5 * v / prm.lambda_par * omm
        dD = -mu * v / prm.lambda_par
    rb = _philox(n, pid, 0, 0, prm.seed, prm.set_id)
    amp, ang = torch.sqrt(-2 * torch.log(_u(rb[0]))), 2 * math.pi * _u(rb[1])
    mudot = 0.5 * omm * (v * divb + mu * divv - 3 * mu * bbgv - 2 / v * bdvdt)
    mun = mu + (mudot + dD) * prm.dt + torch.sqrt(2 * D * prm.dt) * amp * torch.cos(ang)
    mun = torch.where(mun > 1, 2 - mun, mun)
    mun = torch.where(mun < -1, -2 - mun, mun).clamp(-1, 1)
    u = V + (mu * v)[:, None] * b
    noise = 0.0
    if prm.lambda_perp > 0:
        kap = v * prm.lambda_perp / 3
        if prm.kappa_drift:
            cth, sth, cph, sph = z / r, rho / r, x / rho, y / rho
            br = (b[:, 0] * cph + b[:, 1] * sph) * sth + b[:, 2] * cth
            bt = ((b[:, 0] * cph + b[:, 1] * sph) * cth - b[:, 2] * sth) / r
            bp = (b[:, 1] * cph - b[:, 0] * sph) / rho
            g3 = dB[0] * br[:, None] + dB[1] * bt[:, None] + dB[2] * bp[:, None]
            par = (b * g3).sum(1, keepdim=True)
            u = u - kap[:, None] * (divb[:, None] * b + (g3 - b * par) / Bm[:, None])
        cz, cx = torch.hypot(b[:, 0], b[:, 1]), torch.hypot(b[:, 1], b[:, 2])
        zero = torch.zeros_like(cz)
        e1 = torch.where((cz >= 0.1)[:, None], torch.stack((b[:, 1] / cz, -b[:, 0] / cz, zero), 1),
                         torch.stack((zero, b[:, 2] / cx, -b[:, 1] / cx), 1))
        e2 = torch.linalg.cross(b, e1)
        z2 = torch.sqrt(-2 * torch.log(_u(rb[2]))) * torch.cos(2 * math.pi * _u(rb[3]))
        noise = torch.sqrt(2 * kap * prm.dt)[:, None] * ((amp * torch.sin(ang))[:, None] * e1 + z2[:, None] * e2)
    new = torch.stack((x, y, z), 1) + u * prm.dt + noise
    pdot = 0.5 * (1 - 3 * mu * mu) * bbgv - 0.5 * omm * divv - mu / v * bdvdt
    pn = p * (torch.exp(pdot * prm.dt) if prm.p_update == "exp" else 1 + pdot * prm.dt)
    return dict(x=new[:, 0], y=new[:, 1], z=new[:, 2], mu=mun, p=pn, w=q["w"]), (r, th, ph)


def _energy(p):
    return MC2 * p * p / (torch.sqrt(1 + p * p) + 1)


def _exact_tally(obs, t, q, rtp, S, S2, cls, pid, dt):
    r, th, ph = rtp
    off = 0
    for o in obs:
        it = math.floor((t - o.t_lo) * o.nt / (o.t_hi - o.t_lo))
        here, off = off, off + o.ne * o.nt
        if not 0 <= it < o.nt:
            continue
        if o.kind == "slab":
            inside = (q["x"] - o.r).abs() <= o.dr
        else:
            inside = (r - o.r).abs() <= o.dr
        if o.kind in ("box", "ring"):
            inside &= (th - o.th).abs() <= o.dth
        if o.kind == "box":
            inside &= (torch.remainder(ph - o.ph + math.pi, 2 * math.pi) - math.pi).abs() <= o.dph
        le = torch.log(_energy(q["p"]) / o.e_lo) * (o.ne / math.log(o.e_hi / o.e_lo))
        inside &= (le >= 0) & (le < o.ne)
        k = inside.nonzero()[:, 0]
        col = (ph[k] * o.nt / (2 * math.pi)).long().clamp(max=o.nt - 1) if o.kind == "ring" else it
        b = here + le[k].long() * o.nt + col
        w = q["w"][k] * dt
        S.index_add_(0, b, w)
        S2.index_add_(0, b, w * w)
        cls.view(-1).index_add_(0, b * 32 + pid[k] % 32, w)


#: Steps up to which the 64-bit run is made: beyond a few hundred steps the
#: pitch-angle map (whose drift jumps, or diverges, at mu = 0) has carried any rounding
#: difference to the size of mu itself, and a 64-bit path says nothing about a 32-bit one.
EXACT_STEPS = 400


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("advance", "adjoint") or case["steps"] > EXACT_STEPS or case["n"] > 150_000 or \
            (kind == "adjoint" and case["autograd"]):
        return None                        # conversions give bytes; long and large runs: see above
    g, prm = _grid(case), _params(case, seed)
    fields = _exact_fields(case, seed)
    q, pid = _exact_inject(case, seed, fields)
    I = 1.0 if prm.dmumu == "iso" else _norm(prm)
    alive = torch.ones(case["n"], dtype=torch.bool, device="cuda")
    out = {k: v.clone() for k, v in q.items()}
    injected = float(q["w"].sum())
    absorbed = [0.0] * 8
    if kind == "adjoint":
        ob = _smooth(case)
        Ji = torch.zeros(case["n"], dtype=F64, device="cuda")
    else:
        obs = _observers(case)
        nb = sum(o.ne * o.nt for o in obs)
        S, S2 = torch.zeros(nb, dtype=F64, device="cuda"), torch.zeros(nb, dtype=F64, device="cuda")
        cls = torch.zeros((1, nb, 32), dtype=F64, device="cuda")
    for n in range(case["steps"]):
        k = alive.nonzero()[:, 0]
        if k.numel() == 0:
            break
        cur = {a: v[k] for a, v in out.items()}
        new, rtp = _exact_step(case, g, prm, I, fields, n, k, cur)
        t = prm.t0 + n * prm.dt
        if kind == "adjoint":
            a = (rtp[0] - ob.r_o) / ob.sigma_r
            b = torch.log(_energy(cur["p"]) / ob.e_c) / ob.sigma_lnE
            c = (t - ob.t_c) / ob.sigma_t
            Ji[k] += cur["w"] * prm.dt * torch.exp(-0.5 * (a * a + b * b + c * c))
        else:
            _exact_tally(obs, t, cur, rtp, S, S2, cls, k, prm.dt)
        for a, v in new.items():
            out[a][k] = v
        rn = torch.sqrt(new["x"] ** 2 + new["y"] ** 2 + new["z"] ** 2)
        inner, outer = rn < g.r_min, rn > g.r_max
        theta = ((new["z"] > rn * math.cos(g.th_min)) | (new["z"] < rn * math.cos(g.th_max))) & ~inner & ~outer
        for slot, gone in ((1, inner), (2, outer), (3, theta)):
            absorbed[slot] += float(new["w"][gone].sum())
        alive[k[inner | outer | theta]] = False
    out.update(id=None, status=None)
    if case["wind"] == "parker":
        out["z"] = None                    # injected at theta = 90 deg, z is the rounding of cos(pi / 2)
    if kind == "adjoint":
        # the gradients are those of a hybrid pathwise / score estimator that only the library defines
        return {"J": Ji.sum(), "J_i": Ji, "grad": None, "per_particle": None, **out}
    absorbed[0] = injected
    return {**out, "S": S, "S2": S2, "C": None, "S_class": cls,
            "ledger_w": torch.tensor(absorbed, dtype=F64), "ledger_n": None}
