"""Timed cases of the strong-field QED Monte Carlo step: what a user of libsfq has it do,
through the public binding (`paper_2301_07684_gb300.sfq`, `batch`, `cascade`).

Every case is a dict of plain values; `prepare` makes what a program has in hand (beams,
fields, buffers, contexts, trained networks), `run` is one pass, and `exact` restates the
pass in binary64 with plain torch where that has a value.  A pass of a stepping case starts
from the beam it was given: the population is copied into the working buffers, stepped, and
its state returned.

Product records are an unordered set (the step appends them with atomics), so the cases
that return them sort them first, as the library's own runs do (`sort_products`); the
others return the stepped state, which every record was taken from, and the counters.
Populations that grow on the device are returned in the order of their ids.
"""
import math

import numpy as np
import torch

from paper_2301_07684_gb300 import batch, cascade, sfq
from paper_2301_07684_gb300 import workloads as W

DEV = "cuda"
SEED = 12345                       # key of the Monte Carlo draws (Philox)
EXACT_SAMPLES = 20000              # most elements of the samplers that exact() inverts
EXACT_UPDATES = 5000000            # most particle-steps that exact() replays


def listed():
    return [
        # Rates and one energy sample of a handful of particles, binary64: the library called
        # as a function, where launches and the binding are what a caller waits for.
        dict(name="tables_f64_4k", path="tables", n=4096, precision="fp64"),
        # The same entry points over a whole population in binary32.
        dict(name="tables_f32_16m", path="tables", n=1 << 24, precision="fp32"),
        # A particle-in-cell code's loop at production size: fields interpolated to the
        # particles in six arrays, a new set every step, one Monte Carlo step each.
        dict(name="pic_f32_16m", path="pic", n=1 << 24, steps=8, precision="fp32", push=False, sort=False),
        # The same loop on one rank's small, odd-sized share, its photons sorted with the
        # scratch-free sort at the end.
        dict(name="pic_f32_10k", path="pic", n=10007, steps=16, precision="fp32", push=False, sort=True),
        # The plain binary64 path, coupled to the Boris push, records sorted.
        dict(name="pic_push_f64_1m", path="pic", n=1200003, steps=4, precision="fp64", push=True, sort=True),
        # The analytic plane wave, the steps recorded into one CUDA graph.
        dict(name="wave_graph_f32_4m", path="wave", n=4194304 + 77, steps=40, fused=False, precision="fp32"),
        # The same field with all steps fused into one launch.
        dict(name="wave_fused_f32_1m", path="wave", n=1 << 20, steps=100, fused=True, precision="fp32"),
        # Many beams of uneven size and mixed species in one launch, pairs stepped as
        # children, one graph, records sorted by (parent id, step).
        dict(name="beams_f32_64", path="beams", beams=64, scale=0.0625, steps=40, precision="fp32"),
        # Pair creation by photons, the pairs stepped by the beyond-LCFA model.
        dict(name="pairs_blcfa_f32_1m", path="pairs", n=1 << 20, steps=40, precision="fp32"),
        # Full cascade: every product is stepped again, the dead compacted away at the end.
        dict(name="cascade_f32_64k", path="cascade", n=1 << 16, steps=80, precision="fp32"),
        # The learned photon sampler over a population, with and without its fallback cells.
        dict(name="surrogate_photon_10m", path="surrogate", kind="photon", n=10000019),
        # Its training: one full-batch loss and gradient, then minibatch steps.
        dict(name="surrogate_train", path="train", kind="photon", n=65541, steps=50, batch=8192),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi], odd as often as even."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["tables", "pic", "pic", "wave", "beams", "pairs", "cascade", "surrogate", "train"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    if path == "tables":
        return dict(path=path, n=_log_int(rng, 1000, 1 << 24 if prec == "fp32" else 1 << 21), precision=prec)
    if path == "pic":
        n = _log_int(rng, 1000, 1 << 23 if prec == "fp32" else 1 << 20)
        return dict(path=path, n=n, steps=rng.randint(2, 10), precision=prec, push=rng.random() < 0.5,
                    sort=n <= 4000000)
    if path == "wave":
        return dict(path=path, n=_log_int(rng, 1000, 1 << 21 if prec == "fp32" else 1 << 17),
                    steps=rng.randint(5, 60), fused=rng.random() < 0.5, precision=prec)
    if path == "beams":
        return dict(path=path, beams=rng.randint(2, 64), scale=math.exp(rng.uniform(math.log(1 / 1024), math.log(1 / 16))),
                    steps=rng.randint(5, 40), precision="fp32")
    if path == "pairs":
        return dict(path=path, n=_log_int(rng, 1000, 1 << 20), steps=rng.randint(5, 40), precision="fp32")
    if path == "cascade":
        return dict(path=path, n=_log_int(rng, 500, 1 << 16), steps=rng.randint(10, 60), precision="fp32")
    kind = rng.choice(["photon", "pair"])
    if path == "surrogate":
        return dict(path=path, kind=kind, n=_log_int(rng, 1000, 10000000))
    return dict(path=path, kind=kind, n=_log_int(rng, 1000, 65536), steps=rng.randint(5, 50),
                batch=64 * rng.randint(16, 128))


# --- inputs -------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _log_uniform(g, n, lo, hi):
    return torch.exp(_uniform(g, n, math.log(lo), math.log(hi)))


def _draw_grid(g, n):
    """The uniforms of the step: odd multiples of 2^-24, exact in both precisions."""
    return (torch.randint(0, 1 << 23, (n,), generator=g, device=DEV).double() + 0.5) * 2.0 ** -23


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _context(case):
    return sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=case.get("precision", "fp32"), seed=SEED)


def _beam(g, n, dtype, gamma0, spread_t):
    """Leptons head-on with the wave: gamma ~ N(gamma0, 5 %), a little divergence; one in
    ten a positron; optical depths of a beam under way, one in ten not yet drawn."""
    gam = gamma0 * (1 + 0.05 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    py = spread_t * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    pz = spread_t * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    px = -torch.sqrt(torch.clamp(gam * gam - 1 - py * py - pz * pz, min=1.0))
    tau = -torch.log(_draw_grid(g, n))
    tau = torch.where(_uniform(g, n) < 0.1, torch.full_like(tau, -1.0), tau)
    species = (_uniform(g, n) < 0.1).to(torch.uint8)                    # 0 electron, 1 positron
    flags = (species << sfq.SFQ_SPECIES_SHIFT) | sfq.SFQ_ALIVE
    return [px.to(dtype), py.to(dtype), pz.to(dtype), tau, flags]


def _fields_of_step(g, k0, step, table, dtype):
    """Six field components at the particles: the wave (a0 = 100) and 1 % of disorder."""
    n = k0.numel()
    f = 100.0 * table[(k0 + step * W.K_STEP) % table.numel()].double()
    noise = lambda: 1.0 * torch.randn(n, generator=g, device=DEV, dtype=torch.float32)
    return [t.to(dtype) for t in (noise(), f + noise(), noise(), noise(), noise(), f + noise())]


# --- prepare --------------------------------------------------------------------------
def prepare(case, seed):
    return globals()["_prepare_" + case["path"]](case, seed)


def _prepare_tables(case, seed):
    g, n, dt = _gen(seed), case["n"], _dtype(case)
    return dict(case=case, ctx=_context(case),
                gamma_e=_log_uniform(g, n, 10.0, 1e4).to(dt), chi_e=_log_uniform(g, n, 1e-3, 100.0).to(dt),
                gamma_g=_log_uniform(g, n, 1e2, 1e5).to(dt), chi_g=_log_uniform(g, n, 0.1, 100.0).to(dt),
                ids=torch.arange(n, device=DEV, dtype=torch.int64) + seed * 1000003)


def _inputs_pic(case, seed):
    g, n, dt = _gen(seed), case["n"], _dtype(case)
    beam = _beam(g, n, dt, 2000.0, 10.0)
    table = torch.as_tensor(W.cos_table(np.float64), device=DEV)
    k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device=DEV)
    return beam, [_fields_of_step(g, k0, s, table, dt) for s in range(case["steps"])]


def _products(capacity, dtype):
    out = sfq.ProductBuffers(capacity, dtype, DEV)
    for t in (out.px, out.py, out.pz, out.parent_id, out.step, out.meta):
        t.zero_()
    return out


def _prepare_pic(case, seed):
    beam, slabs = _inputs_pic(case, seed)
    n, dt = case["n"], _dtype(case)
    out = _products(int(0.09 * n * case["steps"]) + 4096, dt)
    return dict(case=case, ctx=_context(case), beam=beam,
                P=sfq.ParticleBuffers(*[t.clone() for t in beam]), F=[sfq.FieldSource.soa(*s) for s in slabs],
                out=out, counters=sfq.counters_tensor(),
                scratch=torch.empty(sfq.sort_scratch_bytes(out.capacity), dtype=torch.uint8, device=DEV)
                if case["sort"] and out.capacity > sfq.SORT_NOALLOC_MAX_N else None)


def _prepare_wave(case, seed):
    g, n, dt = _gen(seed), case["n"], _dtype(case)
    beam = _beam(g, n, dt, 2000.0, 10.0)
    k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device=DEV, dtype=torch.int32)
    table = torch.as_tensor(W.cos_table(np.float64 if dt == torch.float64 else np.float32), device=DEV)
    return dict(case=case, ctx=_context(case), beam=beam, P=sfq.ParticleBuffers(*[t.clone() for t in beam]),
                F=sfq.FieldSource.plane_wave(k0, table, W.K_STEP, amp0=100.0),
                out=_products(int(0.09 * n * case["steps"]) + 4096, dt),
                counters=sfq.counters_tensor())


def _prepare_beams(case, seed):
    """Beams of one machine setup (counts, species, a0 and gamma0 by the case alone), their
    particles by the seed."""
    ctx, g, nb = _context(case), _gen(seed), case["beams"]
    setup = np.random.default_rng(nb)
    counts = np.maximum(1, np.exp(setup.uniform(math.log(1e3), math.log(4e6), nb)) * case["scale"]).astype(np.int64)
    dev = lambda a: torch.repeat_interleave(torch.as_tensor(a, device=DEV), torch.as_tensor(counts, device=DEV))
    species = dev(np.arange(nb) % 3 if nb < 3 else setup.permutation(np.arange(nb) % 3))
    a0 = dev(setup.uniform(10.0, 300.0, nb))
    gam = dev(np.exp(setup.uniform(math.log(200.0), math.log(1e4), nb)))
    n = int(counts.sum())
    gam = gam * (1 + 0.05 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    px = -torch.where(species == sfq.SFQ_PHOTON, gam, torch.sqrt(gam * gam - 1))
    flags = ((species << sfq.SFQ_SPECIES_SHIFT) | sfq.SFQ_ALIVE).to(torch.uint8)
    k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device=DEV)
    host = lambda t, dt: t.cpu().numpy().astype(dt)
    zero = np.zeros(n, np.float32)
    run_ = batch.BatchRun(ctx, dict(px=host(px, np.float32), py=zero, pz=zero, tau=np.full(n, -1.0),
                                    flags=host(flags, np.uint8), k0=host(k0, np.uint32), amp=host(a0, np.float32),
                                    table=W.cos_table(), k_step=W.K_STEP),
                          products_cap=0, children_cap=n + 64)
    run_.out = _products(int(0.1 * n * case["steps"]) + 4096, torch.float32)
    beam = [t.clone() for t in (run_.P.px, run_.P.py, run_.P.pz, run_.P.tau, run_.P.flags)]
    return dict(case=case, ctx=ctx, run=run_, P=run_.P, beam=beam, sorted=[torch.zeros_like(t) for t in _columns(run_.L)],
                scratch=torch.empty(sfq.sort_scratch_bytes(run_.out.capacity), dtype=torch.uint8, device=DEV))


def _prepare_pairs(case, seed):
    g, n = _gen(seed), case["n"]
    chi_peak, gam = _log_uniform(g, n, 0.1, 100.0), _log_uniform(g, n, 1e2, 1e5)
    z = lambda: torch.zeros(n, device=DEV)
    flags = torch.full((n,), sfq.SFQ_ALIVE | (sfq.SFQ_PHOTON << sfq.SFQ_SPECIES_SHIFT), dtype=torch.uint8, device=DEV)
    beam = [(-gam).float(), z(), z(), torch.full((n,), -1.0, dtype=torch.float64, device=DEV), flags]
    table = torch.as_tensor(W.cos_table(), device=DEV)
    k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device=DEV, dtype=torch.int32)
    amp = (chi_peak * W.RHO / (2.0 * gam)).float()
    cap = 2 * n + 64                                       # a photon converts at most once
    col = lambda dt=torch.float32: torch.zeros(cap, dtype=dt, device=DEV)
    count = torch.zeros(2, dtype=torch.int64, device=DEV)
    L = sfq.ParticleBuffers(col(), col(), col(), col(torch.float64), col(torch.uint8), ids=col(torch.int64),
                            fprev=[col() for _ in range(3)], dfprev=[col() for _ in range(3)],
                            lepton_model=sfq.SFQ_LEPTON_BLCFA_LOCAL, n_dev=count)
    lk0, lamp = col(torch.int32), col()
    spawn = sfq.SpawnBuffers(L, k0=lk0, amp=lamp)
    spawn.count = count
    return dict(case=case, ctx=_context(case), beam=beam, P=sfq.ParticleBuffers(*[t.clone() for t in beam]),
                F=sfq.FieldSource.plane_wave(k0, table, W.K_STEP, amp=amp), L=L,
                FL=sfq.FieldSource.plane_wave(lk0, table, W.K_STEP, amp=lamp), spawn=spawn, spawn_count=count,
                sorted=[torch.zeros_like(t) for t in _columns(L)],
                out=_products(n * case["steps"] // 2 + 4096, torch.float32),
                counters=sfq.counters_tensor())


def _prepare_cascade(case, seed):
    ctx, n = _context(case), case["n"]
    d = W.config2(n=n, seed=seed, a0=150.0, gamma0=1e4)
    run_ = cascade.CascadeRun(ctx, d, capacity=64 * n, products_cap=20 * n)
    A = run_.A
    return dict(case=case, ctx=ctx, run=run_, n=n, sorted=[torch.zeros_like(t) for t in _columns(A.P)],
                beam=[t[:n].clone() for t in (A.P.px, A.P.py, A.P.pz, A.P.tau, A.P.flags, A.P.ids, A.k0)],
                live=A.count.clone())


_NETS = {}


def _network(kind):
    """Weights of a photon or pair surrogate, fitted once per process with plain torch to the
    fitted sampler's own values: what a program loads from its file of trained networks."""
    if kind in _NETS:
        return _NETS[kind]
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=SEED)
    net = sfq.Surrogate(ctx, seed=7, kind=kind)
    g, n = _gen(2024), 1 << 20
    lo, hi = (1e-3, 100.0) if kind == "photon" else (0.1, 100.0)
    chi, u = _log_uniform(g, n, lo, hi).float(), _draw_grid(g, n).float()
    y = net.plain_targets(chi, u) - torch.log(u)
    ok = torch.isfinite(y)
    x, y = _features(chi, u, kind).float()[ok], y[ok]
    shapes = [(64, 2), (64, 64), (64, 64), (1, 64)]
    par = []
    for o, i in shapes:
        for shape in ((o, i), (o,)):
            par.append(((torch.rand(shape, generator=g, device=DEV) * 2 - 1) / math.sqrt(i)).requires_grad_())
    opt = torch.optim.Adam(par, lr=5e-3, fused=True)
    steps = 2500
    for t in range(steps):
        for group in opt.param_groups:
            group["lr"] = 2.5e-3 * (1 + math.cos(math.pi * t / steps)) + 1e-5
        k = torch.randint(0, y.numel(), (8192,), generator=g, device=DEV)
        h = x[k]
        for layer in range(3):
            h = torch.nn.functional.silu(torch.addmm(par[2 * layer + 1], h, par[2 * layer].t()))
        loss = (torch.addmm(par[7], h, par[6].t())[:, 0] - y[k]).square().mean()
        opt.zero_grad(set_to_none=True)
        loss.backward()
        opt.step()
    _NETS[kind] = torch.cat([p.detach().reshape(-1) for p in par]).cpu().numpy()
    net.close()
    ctx.close()
    return _NETS[kind]


def _features(chi, u, kind):
    chi, u = chi.double(), u.double()
    lo, hi = (math.log(1e-3), math.log(100.0)) if kind == "photon" else (math.log(0.1), math.log(100.0))
    return torch.stack([(torch.log(chi) - 0.5 * (lo + hi)) / (0.5 * (hi - lo)), -torch.log1p(-u) / 8 - 1], 1)


def _draws_surrogate(case, seed):
    g, n = _gen(seed), case["n"]
    chi = _log_uniform(g, n, 1e-3 if case["kind"] == "photon" else 0.1, 100.0).float()
    return chi.clamp(1.0001e-3 if case["kind"] == "photon" else 0.10001, 99.99), _draw_grid(g, n).float()


def _prepare_surrogate(case, seed):
    ctx = _context(case)
    net = sfq.Surrogate(ctx, seed=7, kind=case["kind"])
    net.set_params(_network(case["kind"]))
    net.calibrate(3e-3)
    chi, r = _draws_surrogate(case, seed)
    return dict(case=case, ctx=ctx, net=net, chi=chi, r=r, counters=sfq.counters_tensor())


def _inputs_train(case, seed):
    g, n = _gen(seed), case["n"]
    chi = _log_uniform(g, n, 1e-3 if case["kind"] == "photon" else 0.1, 100.0).float()
    u = (_draw_grid(g, n) if case["kind"] == "photon" else (2 * _draw_grid(g, n) - 1).abs().clamp(min=1e-3)).float()
    lim = 1 / np.sqrt(np.concatenate([np.full(192, 2.0), np.full(8577 - 192, 64.0)]))
    theta = (np.random.default_rng(seed).uniform(-1, 1, 8577) * lim).astype(np.float32)
    return chi, u, theta


def _prepare_train(case, seed):
    chi, u, theta = _inputs_train(case, seed)
    ctx = _context(case)
    net = sfq.Surrogate(ctx, seed=7, kind=case["kind"])
    return dict(case=case, ctx=ctx, net=net, chi=chi, u=u, theta=theta, lnw=net.plain_targets(chi, u))


# --- run ------------------------------------------------------------------------------
def run(state):
    return globals()["_run_" + state["case"]["path"]](state)


def _run_tables(s):
    ctx = s["ctx"]
    u = ctx.uniforms(s["ids"], step=3)
    r = u[:, 1].contiguous()
    xi, xi_c = ctx.sample_photon_xi(s["chi_e"], r)
    xe, xp = ctx.sample_pair_xi(s["chi_g"], r)
    return dict(u=u, photon_rate=ctx.photon_rate(s["gamma_e"], s["chi_e"]),
                pair_rate=ctx.pair_rate(s["gamma_g"], s["chi_g"]), xi=xi, xi_c=xi_c, xe=xe, xp=xp)


def _load(P, beam):
    for dst, src in zip((P.px, P.py, P.pz, P.tau, P.flags), beam):
        dst.copy_(src)


def _state(P):
    return dict(px=P.px, py=P.py, pz=P.pz, tau=P.tau, flags=P.flags)


def _records(out):
    """The whole buffers: past the count they hold the zeros they were made with."""
    return dict(px=out.px, py=out.py, pz=out.pz, parent_id=out.parent_id, step=out.step, meta=out.meta)


def _run_pic(s):
    ctx, P, out, case = s["ctx"], s["P"], s["out"], s["case"]
    _load(P, s["beam"])
    out.reset()
    s["counters"].zero_()
    for k, F in enumerate(s["F"]):
        if case["push"]:
            ctx.push(P, F, k, W.DT)
        ctx.mc_step(P, F, k, out, counters=s["counters"])
    got = dict(state=_state(P), counters=s["counters"], count=out.count)
    if case["sort"]:
        n = min(out.n(), out.capacity)
        if n <= sfq.SORT_NOALLOC_MAX_N:
            ctx.sort_products_noalloc(out, n)
        else:
            ctx.sort_products(out, n, s["scratch"])
        got["records"] = _records(out)
    return got


def _run_wave(s):
    ctx, P, out, case = s["ctx"], s["P"], s["out"], s["case"]
    _load(P, s["beam"])
    out.reset()
    s["counters"].zero_()
    if case["fused"]:
        ctx.mc_run_fused(P, s["F"], 0, case["steps"], out, counters=s["counters"])
    else:
        ctx.mc_run(P, s["F"], 0, case["steps"], out, counters=s["counters"])
    return dict(state=_state(P), counters=s["counters"], count=out.count)


def _columns(P):
    return [P.ids, P.px, P.py, P.pz, P.tau, P.flags] + list(P.fprev or []) + list(P.dfprev or [])


def _by_id(P, n, into, tagged=True):
    """The first n particles of a population grown on the device, ordered by (id, tag), in
    the buffers `into`, which past n hold the zeros they were made with."""
    tag = (P.flags[:n] >> sfq.SFQ_TAG_SHIFT).long() & 3
    order = torch.argsort(P.ids[:n] * 4 + tag if tagged else P.ids[:n])
    for src, dst in zip(_columns(P), into):
        torch.index_select(src[:n], 0, order, out=dst[:n])
    return into


def _run_beams(s):
    b = s["run"]
    _load(b.P, s["beam"])
    b.spawn_count.zero_()
    b.out.reset()
    b.counters.zero_()
    b.run(0, s["case"]["steps"])
    n = min(b.out.n(), b.out.capacity)
    s["ctx"].sort_products(b.out, n, s["scratch"])
    return dict(state=_state(b.P), children=_by_id(b.L, b.n_children(), s["sorted"]), records=_records(b.out),
                counters=b.counters)


def _run_pairs(s):
    _load(s["P"], s["beam"])
    s["spawn_count"].zero_()
    s["out"].reset()
    s["counters"].zero_()
    s["ctx"].mc_run(s["P"], s["F"], 0, s["case"]["steps"], s["out"], children=s["L"], children_fields=s["FL"],
                    spawn=s["spawn"], counters=s["counters"])
    n = min(int(s["spawn_count"][0]), s["L"].n)
    return dict(state=_state(s["P"]), leptons=_by_id(s["L"], n, s["sorted"]), counters=s["counters"], count=s["out"].count)


def _run_cascade(s):
    r, n = s["run"], s["n"]
    A = r.A
    for dst, src in zip((A.P.px, A.P.py, A.P.pz, A.P.tau, A.P.flags, A.P.ids, A.k0), s["beam"]):
        dst[:n].copy_(src)
    A.count.copy_(s["live"])
    r.out.reset()
    r.counters.zero_()
    r.run(0, s["case"]["steps"])
    m = r.compact()
    return dict(population=_by_id(r.P, m, s["sorted"], False), counters=r.counters, count=r.out.count)


def _run_surrogate(s):
    s["counters"].zero_()
    sample = s["net"].sample_photon_xi if s["case"]["kind"] == "photon" else s["net"].sample_pair_xi
    net = sample(s["chi"], s["r"], use_flags=False)
    safe = sample(s["chi"], s["r"], use_flags=True, counters=s["counters"])
    return dict(net=list(net), safe=list(safe), counters=s["counters"])


def _run_train(s):
    net, case = s["net"], s["case"]
    net.set_params(s["theta"])
    loss, grad = net.loss_grad(s["chi"], s["u"], s["lnw"])
    hist = net.train(s["chi"], s["u"], s["lnw"], case["steps"], batch=case["batch"], lr=3e-3, seed=9, history=True)
    return dict(loss=loss, grad=grad, history=hist, params=net.get_params())


# --- work -----------------------------------------------------------------------------
def work(case):
    """Bytes read and written once and the operations of the method, by the laws of the
    inputs: about 0.06 photons per lepton and step at a0 = 100, and so on."""
    e = 8 if case.get("precision") == "fp64" else 4
    rec = 3 * e + 13                                   # a product record
    path, n = case["path"], case.get("n", 0)
    if path == "tables":
        return {"bytes": n * (8 + 4 * e + 10 * e), "flops": n * (2 * 30 + 2 * 2 * (81 if e == 4 else 144))}
    if path in ("pic", "wave"):
        k = case["steps"]
        load = n * 2 * (3 * e + 9)                     # the beam into the working buffers
        ev = 0.06 * (3 * e + rec)                      # a recoil and a record
        once = 3 * e + 8 + 1
        if path == "pic":
            push = (3 * e + 1 + 6 * e + 3 * e) if case["push"] else 0
            sort = 0.06 * 2 * rec if case["sort"] else 0
            per = once + 6 * e + 8 + ev + push + sort
        elif case["fused"]:
            load += n * (2 * once + 4)                 # the state once in and once out of the launch
            per = 0.06 * rec
        else:
            per = once + 4 + 8 + ev
        return {"bytes": load + n * k * per, "flops": n * k * (90 + 0.06 * 400)}
    if path == "beams":
        n = case["beams"] * 4.8e5 * case["scale"]      # mean of the log-uniform counts
        per = 3 * e + 9 + 8 + 8 + 0.1 * (3 * e + 3 * rec)
        return {"bytes": n * (42 + case["steps"] * per), "flops": n * case["steps"] * 130}
    if path == "pairs":
        k = case["steps"]
        return {"bytes": n * (42 + k * 37 + 0.4 * k * 77 + 0.3 * k * 37), "flops": n * k * (90 + 0.4 * 600)}
    if path == "cascade":
        m = n * case["steps"] * (1 + 0.05 * case["steps"])       # particle-steps of a growing population
        return {"bytes": m * 37 + n * 0.1 * case["steps"] * 66, "flops": m * 110}
    if path == "surrogate":
        return {"bytes": n * 2 * 16, "flops": n * 2 * (2 * (2 * 64 + 2 * 64 * 64 + 64))}
    m = n + case["steps"] * case["batch"]
    return {"bytes": m * 12 + 8577 * 4 * 6 * case["steps"], "flops": m * 3 * 2 * 8448}


# --- exact: the method in binary64, from its defining integrals ---------------------------
# K_2/3 and Ki_1/3 from their integral representations (DLMF 10.32.9), tabulated over ln x
# and interpolated; the rates and cumulative spectra by Gauss-Legendre panels (Eqs. wtilde,
# wtilde_pair, pe_eff_int_2, tilde_I_pp of arXiv:2301.07684).
_GL = {}


def _gauss(k):
    if k not in _GL:
        x, w = np.polynomial.legendre.leggauss(k)
        _GL[k] = (torch.as_tensor(x, device=DEV), torch.as_tensor(w, device=DEV))
    return _GL[k]


def _lagrange(tab, t):
    """8-point interpolation of tab (rows of values on the integers) at t."""
    i = torch.clamp(torch.floor(t).long() - 3, 0, tab.shape[-1] - 8)
    f = t - i
    out = torch.zeros((tab.shape[0],) + t.shape, dtype=torch.float64, device=DEV)
    for k in range(8):
        c = torch.ones_like(t)
        for j in range(8):
            if j != k:
                c = c * (f - j) / (k - j)
        out += tab[:, i + k] * c
    return out


_LX0, _LX1, _LH = math.log(1e-30), math.log(760.0), 0.02
_BES = []


def _bessel(x):
    """e^x K_2/3(x) and e^x Ki_1/3(x) = e^x int_x^inf K_1/3 for x in [1e-30, 760]."""
    if not _BES:
        lx = torch.arange(_LX0, _LX1 + 8 * _LH, _LH, dtype=torch.float64, device=DEV)
        t = torch.arange(0, 78, 0.02, dtype=torch.float64, device=DEV)
        wt = torch.full_like(t, 0.02)
        wt[0] = 0.01
        d = torch.exp(lx)[:, None] * (2 * torch.sinh(t / 2) ** 2)            # x (cosh t - 1)
        e = torch.exp(-d) * wt
        k23 = (e * torch.cosh(2 * t / 3)).sum(1)
        ki = (e * torch.cosh(t / 3) / torch.cosh(t)).sum(1)
        _BES.append(torch.stack([torch.log(k23), torch.log(ki)]))
    v = _lagrange(_BES[0], (torch.log(x) - _LX0) / _LH)
    return torch.exp(v[0]), torch.exp(v[1])


def _f_photon(w, chi):
    x = torch.clamp(w ** 3, 1e-30, 750.0)
    k, ki = _bessel(x)
    o = 1 + 1.5 * chi * w ** 3
    return 9 * w * w / (2 * o ** 3) * ((1 + o * o) * k - o * ki) * torch.exp(-x)


def _f_rate_pair(t, chi):                              # v = tanh t in Eq. wtilde_pair
    eta = torch.clamp(8 * torch.cosh(t) ** 2 / (3 * chi), 1e-12, 750.0)
    return (9 - torch.tanh(t) ** 2) / 3 * _bessel(eta)[0] * torch.exp(-eta)


def _f_pair(t, chi):                                   # v = tanh t in Eq. tilde_I_pp
    eta = torch.clamp(8 * torch.cosh(t) ** 2 / (3 * chi), 1e-12, 750.0)
    k, ki = _bessel(eta)
    v2 = torch.tanh(t) ** 2
    return (2 * (1 + v2) * k + (1 - v2) * ki) * torch.exp(-eta)


def _edges(which):
    if which == "photon":
        return torch.cat([torch.zeros(1), 700 ** (1 / 3) * 2.0 ** (-0.5 * torch.arange(24, -1, -1))]).double().to(DEV)
    return torch.arange(0, 9.0 + 1e-9, 0.1, dtype=torch.float64, device=DEV)


def _panels(f, edges, chi):
    """Integral of f over every panel, for every chi."""
    x, w = _gauss(24)
    a, b = edges[:-1], edges[1:]
    node = 0.5 * (a + b)[:, None] + 0.5 * (b - a)[:, None] * x
    out = torch.empty((chi.numel(), a.numel()), dtype=torch.float64, device=DEV)
    for i in range(0, chi.numel(), 512):
        c = chi[i:i + 512, None, None]
        v = f(node[None].expand(c.shape[0], -1, -1), c.expand(-1, *node.shape))
        out[i:i + 512] = (v * w).sum(2) * (0.5 * (b - a))
    return out


_WT = {}


def _wtilde(chi, which):
    """W~_rad or W~_pair by interpolation of their quadratures on a fine grid of ln chi."""
    lo, hi, m = (1e-9, 200.0, 2600) if which == "photon" else (0.09, 200.0, 1600)
    if which not in _WT:
        grid = torch.exp(torch.linspace(math.log(lo), math.log(hi), m, dtype=torch.float64, device=DEV))
        f, e = (_f_photon, _edges("photon")) if which == "photon" else (_f_rate_pair, _edges("pair"))
        _WT[which] = torch.log(_panels(f, e, grid).sum(1))[None]
    t = (torch.log(chi.clamp(lo, hi)) - math.log(lo)) / (math.log(hi) - math.log(lo)) * (m - 1)
    return torch.exp(_lagrange(_WT[which], t)[0])


def _invert(which, chi, r):
    """The root w of I~_pe(w, chi) = r W~, or t (v = tanh t) of I~_pp = r W~_pair; the upper
    half is solved in the complementary form, which keeps the precision of the tail."""
    f, edges = (_f_photon if which == "photon" else _f_pair), _edges(which)
    I = _panels(f, edges, chi)
    tot = I.sum(1)
    lower = torch.cat([torch.zeros_like(tot)[:, None], I.cumsum(1)], 1)          # up to each edge
    upper = torch.cat([I.flip(1).cumsum(1).flip(1), torch.zeros_like(tot)[:, None]], 1)
    up = r >= 0.5
    goal = torch.where(up, (1 - r) * tot, r * tot)
    below = torch.where(up[:, None], upper >= goal[:, None], lower <= goal[:, None])
    p = (below.long().sum(1) - 1).clamp(0, I.shape[1] - 1)
    at = lambda m, q: m.gather(1, q[:, None])[:, 0]
    a, b = edges[p], edges[p + 1]
    base = torch.where(up, at(upper, p + 1), at(lower, p))
    x, w = _gauss(24)
    lo, hi, z = a.clone(), b.clone(), 0.5 * (a + b)
    for _ in range(60):
        s, t = torch.where(up, z, a), torch.where(up, b, z)
        node = 0.5 * (s + t)[:, None] + 0.5 * (t - s)[:, None] * x
        part = (f(node, chi[:, None].expand_as(node)) * w).sum(1) * 0.5 * (t - s)
        g = torch.where(up, goal - base - part, base + part - goal)              # rises with z
        lo, hi = torch.where(g < 0, z, lo), torch.where(g < 0, hi, z)
        step = z - g / f(z, chi).clamp(min=1e-300)
        new = torch.where((step > lo) & (step < hi), step, 0.5 * (lo + hi))
        done = bool(((new - z).abs() <= 4e-16 * z).all())
        z = new
        if done:
            break
    return z


def _photon_s(chi, r):
    w = torch.cat([_invert("photon", c, q) for c, q in zip(chi.split(4096), r.split(4096))])
    return 1.5 * chi * w ** 3


def _pair_shares(chi, r):
    rp = 2 * r - 1
    t = torch.cat([_invert("pair", c, q) for c, q in zip(chi.split(4096), rp.abs().split(4096))])
    small = 1 / (torch.exp(2 * t) + 1)
    return torch.where(rp >= 0, 1 - small, small), torch.where(rp >= 0, small, 1 - small)


def _philox(ids, step, tag):
    """Four 32-bit words per id of Philox4x32-10 (Salmon et al., SC'11), in int64."""
    M = 0xFFFFFFFF

    def mul(a, b):
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        s = p1 + (p0 >> 16)
        return s >> 16, ((s & 0xFFFF) << 16) | (p0 & 0xFFFF)

    c = [ids & M, (ids >> 32) & M, torch.full_like(ids, step), torch.full_like(ids, tag)]
    k = [SEED & M, SEED >> 32]
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & M, (k[1] + 0xBB67AE85) & M]
    return [((v >> 9).double() + 0.5) * 2.0 ** -23 for v in c]


RHO = W.REF_LEN / 3.8615926796e-13
PREF = 7.2973525693e-3 / (math.sqrt(3.0) * math.pi) * RHO


def exact(case, seed):
    f = globals().get("_exact_" + case["path"])
    return f(case, seed) if f else None


def _exact_tables(case, seed):
    s = _prepare_tables(case, seed)
    ge, xe, gg, xg = (s[k].double() for k in ("gamma_e", "chi_e", "gamma_g", "chi_g"))
    got = dict(u=torch.stack(_philox(s["ids"], 3, 0), 1), xi=None, xi_c=None, xe=None, xp=None,
               photon_rate=PREF * xe / ge * torch.cat([_wtilde(c, "photon") for c in xe.split(1 << 20)]),
               pair_rate=PREF / gg * torch.cat([_wtilde(c, "pair") for c in xg.split(1 << 20)]))
    if case["n"] <= EXACT_SAMPLES:
        r = got["u"][:, 1]
        s = _photon_s(xe, r)
        got["xi"], got["xi_c"] = s / (1 + s), 1 / (1 + s)
        got["xe"], got["xp"] = _pair_shares(xg, r)
    return got


def _exact_pic(case, seed):
    n, steps = case["n"], case["steps"]
    if n * steps > EXACT_UPDATES:
        return None
    beam, slabs = _inputs_pic(case, seed)
    p = [t.double() for t in beam[:3]]
    tau, flags = beam[3].clone(), beam[4]
    ids = torch.arange(n, device=DEV)
    dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]
    cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]
    q = torch.where(((flags >> sfq.SFQ_SPECIES_SHIFT) & 3) == sfq.SFQ_ELECTRON, -1.0, 1.0).double()
    alive = torch.ones(n, dtype=torch.bool, device=DEV)
    rec = []
    for k, slab in enumerate(slabs):
        E, B = [t.double() for t in slab[:3]], [t.double() for t in slab[3:]]
        if case["push"]:
            u = [a + 0.5 * q * W.DT * e for a, e in zip(p, E)]
            t = [0.5 * q * W.DT / torch.sqrt(1 + dot(u, u)) * b for b in B]
            v = [a + c for a, c in zip(u, cross(u, t))]
            sv = [2 * c / (1 + dot(t, t)) for c in t]
            new = [a + c + 0.5 * q * W.DT * e for a, c, e in zip(u, cross(v, sv), E)]
            p = [torch.where(alive, a, b) for a, b in zip(new, p)]
        gam = torch.sqrt(1 + dot(p, p))
        F = [gam * e + c for e, c in zip(E, cross(p, B))]
        chi = torch.sqrt(torch.clamp(dot(F, F) - dot(p, E) ** 2, min=0.0)) / RHO
        d = PREF * W.DT * chi / gam * _wtilde(chi, "photon")
        w = _philox(ids, k, 0)
        tau = torch.where(alive, torch.where(tau < 0, -torch.log(w[3]), tau) - d, tau)
        i = torch.nonzero((tau < 0) & alive)[:, 0]
        tau[i] = -torch.log(w[0][i])
        s = _photon_s(chi[i], w[1][i])
        pm, g = torch.sqrt(dot(p, p))[i], gam[i]
        new = torch.sqrt(torch.clamp((g / (1 + s)) ** 2 - 1, min=0.0))
        dirs = [a[i] / pm for a in p]
        rec.append([i] + [a * g * s / (1 + s) for a in dirs])
        for a, c in zip(p, dirs):
            a[i] = c * new
        alive[i] = new > 0
    got = dict(state=dict(px=p[0], py=p[1], pz=p[2], tau=tau, flags=None), counters=None, count=None)
    if case["sort"]:
        order = torch.argsort(torch.cat([r[0] * steps + k for k, r in enumerate(rec)]))
        cols = [torch.zeros(int(0.09 * n * steps) + 4096, dtype=torch.float64, device=DEV) for _ in range(3)]
        for c in range(3):
            cols[c][:order.numel()] = torch.cat([r[1 + c] for r in rec])[order]
        got["records"] = dict(px=cols[0], py=cols[1], pz=cols[2], parent_id=None, step=None, meta=None)
    return got


def _layers(theta):
    at, out = 0, []
    for o, i in [(64, 2), (64, 64), (64, 64), (1, 64)]:
        out.append((theta[at:at + o * i].reshape(o, i), theta[at + o * i:at + o * i + o]))
        at += o * i + o
    return out


def _forward(layers, x):
    for k, (w, b) in enumerate(layers):
        x = x @ w.t() + b
        if k < 3:
            x = torch.nn.functional.silu(x)
    return x[:, 0]


def _exact_surrogate(case, seed):
    """The network alone in 64 bits, with the weights rounded to bfloat16 as they are used."""
    chi, r = (t.double() for t in _draws_surrogate(case, seed))
    theta = torch.as_tensor(_network(case["kind"]), device=DEV)
    layers = [(w.bfloat16().double(), b.double()) for w, b in _layers(theta)]
    u = r if case["kind"] == "photon" else (2 * r - 1).abs()
    y = torch.cat([_forward(layers, _features(c, q, case["kind"])) for c, q in zip(chi.split(1 << 20), u.split(1 << 20))])
    if case["kind"] == "photon":
        s = 1.5 * chi * torch.exp(3 * (y + torch.log(u)))
        return dict(net=[s / (1 + s), 1 / (1 + s)], safe=[None, None], counters=None)
    small = 0.5 * torch.exp(-u * torch.exp(y))
    xe = torch.where(r >= 0.5, 1 - small, small)
    return dict(net=[xe, torch.where(r >= 0.5, small, 1 - small)], safe=[None, None], counters=None)


def _exact_train(case, seed):
    """Loss and gradient by automatic differentiation; the trained weights have no such value."""
    chi, u, theta = _inputs_train(case, seed)
    ctx = _context(case)
    net = sfq.Surrogate(ctx, seed=7, kind=case["kind"])
    lnw = net.plain_targets(chi, u).double()           # the targets are inputs of the training
    net.close()
    ctx.close()
    th = torch.as_tensor(theta, device=DEV).double().requires_grad_()
    ok = torch.isfinite(lnw)
    y = _forward(_layers(th), _features(chi, u, case["kind"]))
    loss = torch.where(ok, y - torch.where(ok, lnw, 0.0) + torch.log(u.double()), 0.0).square().sum() / chi.numel()
    loss.backward()
    return dict(loss=loss.detach().reshape(1), grad=th.grad, history=None, params=None)
