"""Launch rules of the entry points: the sizes at which a kernel or its launch shape changes.
An element's result does not depend on how many elements a call has, so every size is
compared bit for bit with one large call over the same elements."""
import numpy as np
import pytest
import torch

from paper_2301_07684_gb300 import sfq
from paper_2301_07684_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _elements(n, dtype, seed=5):
    g = np.random.default_rng(seed)
    dev = lambda a: torch.as_tensor(a).to(device="cuda", dtype=dtype)
    # the whole range of both samplers and its outside, with the special values at the front
    chi = 10.0 ** g.uniform(-5, 4, n)
    gam = 10.0 ** g.uniform(0, 5, n)
    r = (g.integers(0, 1 << 23, n) + 0.5) / (1 << 23)
    chi[:6] = [0.0, np.nan, -1.0, np.inf, 4096.0, 1e-30]
    r[6:10] = [0.0, 1.0, np.nan, 2.0 ** -24]
    return dev(gam), dev(chi), dev(r)


def _all(ctx, gam, chi, r, ids, counters):
    return [ctx.uniforms(ids, 3, 1), ctx.photon_rate(gam, chi, counters=counters),
            ctx.pair_rate(gam, chi, counters=counters), *ctx.sample_photon_xi(chi, r, counters=counters),
            *ctx.sample_pair_xi(chi, r, counters=counters)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_element_calls_of_every_size_agree(precision):
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=4)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    big = sms * 256 * 9 + 77
    gam, chi, r = _elements(big, ctx.dtype)
    ids = torch.arange(big, device="cuda", dtype=torch.int64)
    whole = _all(ctx, gam, chi, r, ids, None)
    for n in (1, 31, 32, 33, sms * 32 - 1, sms * 32 + 1, 4096, sms * 255 + 1, sms * 256, sms * 256 * 8 + 1):
        part = _all(ctx, gam[:n], chi[:n], r[:n], ids[:n], None)
        for a, b in zip(part, whole):
            assert torch.equal(a.view(torch.uint8), b[:n].contiguous().view(torch.uint8)), n
    # the counters count every element once, whatever the shape
    cnt = [sfq.counters_tensor() for _ in range(2)]
    _all(ctx, gam, chi, r, ids, cnt[0])
    for k in range(0, big, 40000):
        s = slice(k, min(k + 40000, big))
        _all(ctx, gam[s].clone(), chi[s].clone(), r[s].clone(), ids[s].clone(), cnt[1])
    assert sfq.counters_dict(cnt[0]) == sfq.counters_dict(cnt[1])


@pytest.mark.parametrize("k", [9, 8, 7])
def test_sorted_sampler_tiles(k):
    """Binary32 sampler calls sort tiles of 4096 elements once every SM has a tile: the draws
    and counters of calls around that size equal those of calls below it, with the full and
    the truncated tables, with every element in one piece and with an unused second output."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    ctx.set_sampler_coefficients(k)
    line = torch.cuda.get_device_properties(0).multi_processor_count * 4096
    big = 2 * line + 1
    _, chi, r = _elements(big, ctx.dtype, seed=k)
    one = torch.full_like(chi, 1.3), torch.full_like(r, 0.3)
    for x, u in ((chi, r), one):
        cnt = [sfq.counters_tensor() for _ in range(2)]
        parts = [(ctx.sample_photon_xi(x[a:a + 99328], u[a:a + 99328], counters=cnt[0]),
                  ctx.sample_pair_xi(x[a:a + 99328], u[a:a + 99328], counters=cnt[0])) for a in range(0, big, 99328)]
        small = [torch.cat([p[i][j] for p in parts]) for i in (0, 1) for j in (0, 1)]
        for n in (line - 1, line, line + 1, line + 4095, big):
            c = cnt[1] if n == big else None
            whole = [*ctx.sample_photon_xi(x[:n], u[:n], counters=c), *ctx.sample_pair_xi(x[:n], u[:n], counters=c)]
            for a, b in zip(whole, small):
                assert torch.equal(a.view(torch.int32), b[:n].view(torch.int32)), n
        assert sfq.counters_dict(cnt[0]) == sfq.counters_dict(cnt[1])
    xi = torch.empty_like(chi)
    st = sfq.lib().sfq_sample_photon_xi(ctx._h, big, sfq._ptr(chi), sfq._ptr(r), sfq._ptr(xi), None, None, sfq._stream())
    assert st == 0 and torch.equal(xi, ctx.sample_photon_xi(chi, r)[0])


def _sort_keys(kind, n, g):
    """(parent id, step, meta) of one form of records; the step and meta bits that differ and
    the parent-id bits that differ decide the sort's path."""
    meta = np.full(n, 2, np.uint8)                              # a photon of a primary
    step = g.integers(0, 200, n).astype(np.uint32)
    pid = g.integers(0, max(n // 3, 1), n).astype(np.uint64)
    if kind == "pairs":
        member = g.integers(0, 3, n)
        meta = (np.array([2, 0, 1])[member] | member << 2 | g.integers(0, 3, n) << 4 | g.integers(0, 4, n) << 6).astype(np.uint8)
    elif kind == "same":
        step[:], pid[:] = 7, 1 << 40
    elif kind == "offset":                                      # a rank's id range, late steps
        step, pid = step + np.uint32(0xFFFFFF00), pid + np.uint64((1 << 50) + 12345)
    elif kind == "hashed":                                      # a cascade's descendants: 64 bits
        pid = g.integers(0, 1 << 63, n, dtype=np.uint64) * np.uint64(2) + np.uint64(1)
        step = g.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    elif kind.startswith("width"):                              # exactly so many differing bits
        w = int(kind[5:]) - 6                                   # steps 0 .. 3, members and tags: 6 bits
        pid = g.integers(0, 1 << w, n, dtype=np.uint64)
        pid[:2] = 0, (1 << w) - 1
        step = g.integers(0, 4, n).astype(np.uint32)
        meta = (g.integers(0, 64, n)).astype(np.uint8)
        step[:2], meta[:2] = (0, 3), (0, 63)
    return pid, step, meta


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["photons", "pairs", "same", "offset", "hashed", "width32", "width33", "width64",
                                  "width65"])
def test_sort_paths(kind, precision):
    """The one-block sort, the composite keys of 32 and 64 bits and the two stages, at the edges
    of a block's records, of tiles and of the one-block path, against numpy's stable sort of
    every column; the scratch-free call alike."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=4)
    g = np.random.default_rng(len(kind))
    for n in (2, 33, 1023, 1025, 16383, 16384, 16385, 5 * 4096, 5 * 4096 + 1, 300001):
        pid, step, meta = _sort_keys(kind, n, g)
        p = g.standard_normal((3, n))
        order = np.lexsort(((meta >> 4) & 3, (meta >> 2) & 3, step, pid))
        for noalloc in (False, True):
            out = sfq.ProductBuffers(n + 5, ctx.dtype, "cuda")
            for t, a in zip((out.px, out.py, out.pz, out.parent_id, out.step, out.meta),
                            (*p, pid.view(np.int64), step.view(np.int32), meta)):
                t[:n] = torch.as_tensor(a).to(device="cuda", dtype=t.dtype)
                t[n:] = 77
            out.count[0] = n
            (ctx.sort_products_noalloc if noalloc else ctx.sort_products)(out)
            r = out.to_numpy()
            assert all((t[n:] == 77).all() for t in (out.px, out.parent_id, out.step, out.meta))
            assert np.array_equal(r["parent_id"], pid[order]) and np.array_equal(r["step"], step[order]), (n, noalloc)
            assert np.array_equal(r["meta"], meta[order]), (n, noalloc)
            for k, a in zip(("px", "py", "pz"), p):
                assert np.array_equal(r[k], a.astype(r[k].dtype)[order]), (n, noalloc)


@pytest.mark.parametrize("n", [1, 63, 65, 127 * 64, 128 * 64, 128 * 64 + 1, 257 * 64 - 3])
def test_loss_and_gradient_around_the_reduction_chunks(n):
    """Gradient partials are per 64 samples and reduced 128 at a time; against automatic
    differentiation in binary64.  A gradient is a binary32 sum of at most n terms, each a
    chain of 64-term binary32 sums: 2 (64 + 64) 2^-24 = 1.5e-5 relative to the norm covers
    both when the errors add up."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    net = sfq.Surrogate(ctx, seed=3)
    g = np.random.default_rng(n)
    chi = torch.as_tensor(np.exp(g.uniform(np.log(1e-3), np.log(100.0), n)).astype(np.float32)).cuda()
    u = torch.as_tensor(((g.integers(0, 1 << 23, n) + 0.5) / (1 << 23)).astype(np.float32)).cuda()
    lnw = net.plain_targets(chi, u)
    loss, grad = net.loss_grad(chi, u, lnw)
    th = torch.as_tensor(net.get_params()).cuda().double().requires_grad_()
    c, s = 0.5 * (np.log(1e-3) + np.log(100.0)), 0.5 * (np.log(100.0) - np.log(1e-3))
    h = torch.stack([(chi.double().log() - c) / s, -torch.log1p(-u.double()) / 8 - 1], 1)
    at = 0
    for k, (o, i) in enumerate([(64, 2), (64, 64), (64, 64), (1, 64)]):
        h = h @ th[at:at + o * i].view(o, i).t() + th[at + o * i:at + o * i + o]
        h = torch.nn.functional.silu(h) if k < 3 else h
        at += o * i + o
    ref = (h[:, 0] - lnw.double() + u.double().log()).square().mean()
    ref.backward()
    assert abs(float(loss) / float(ref.detach()) - 1) < 1.5e-5
    assert float((grad.double() - th.grad).norm() / th.grad.norm()) < 1.5e-5


@pytest.mark.parametrize("kind", ["photon", "pair"])
def test_surrogate_tiles(kind):
    """The tensor-core kernel takes tiles of 256 draws, two per thread: calls around a tile and
    around one wave of blocks give the draws of a longer call, with and without the flags."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    net = sfq.Surrogate(ctx, seed=3, kind=kind)
    net.calibrate(0.2)                                          # an untrained network: some cells flagged, not all
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 256
    big = 2 * wave + 300
    _, chi, r = _elements(big, torch.float32)
    sample = net.sample_photon_xi if kind == "photon" else net.sample_pair_xi
    for flags in (False, True):
        cnt = [sfq.counters_tensor() for _ in range(2)]
        whole = sample(chi, r, use_flags=flags, counters=cnt[0])
        for n in (1, 127, 128, 129, 255, 256, 257, 511, wave - 1, wave, wave + 1):
            for a, b in zip(sample(chi[:n], r[:n], use_flags=flags), whole):
                assert torch.equal(a.view(torch.int32), b[:n].view(torch.int32)), n
        for k in range(0, big, 70144):
            sample(chi[k:k + 70144], r[k:k + 70144], use_flags=flags, counters=cnt[1])
        assert sfq.counters_dict(cnt[0]) == sfq.counters_dict(cnt[1])
        assert (sfq.counters_dict(cnt[0])["surrogate_fallbacks"] > 0)


def _mixed_population(n, dtype, seed):
    """Electrons, positrons, photons and dead particles in no order, some without an optical
    depth, with the special momenta at the front."""
    g = np.random.default_rng(seed)
    p = np.stack([-10.0 ** g.uniform(0, 4, n), g.normal(0, 10, n), g.normal(0, 10, n)])
    p[:, :4] = [[0.0, np.nan, 1e30, 1e-30]] * 3 if n >= 4 else p[:, :4]
    flags = (g.integers(0, 5, n) > 0).astype(np.uint8) | (g.integers(0, 3, n) << 2).astype(np.uint8)
    flags[n // 3:n // 2] = sfq.SFQ_ALIVE                        # a run of electrons, a run of photons
    flags[n // 2:2 * n // 3] = sfq.SFQ_ALIVE | (sfq.SFQ_PHOTON << 2)
    tau = np.where(g.random(n) < 0.2, -1.0, g.exponential(0.3, n))
    dev = lambda a, dt: torch.as_tensor(a).to(device="cuda", dtype=dt)
    return [dev(a, dtype) for a in p] + [dev(tau, torch.float64), dev(flags, torch.uint8)]


def _run_mixed(ctx, beam, fields, steps, fused=False):
    P = sfq.ParticleBuffers(*[t.clone() for t in beam])
    out, cnt = sfq.ProductBuffers(3 * P.n * steps + 64, ctx.dtype, "cuda"), sfq.counters_tensor()
    if fused:
        ctx.mc_run_fused(P, fields, 0, steps, out, counters=cnt)
    else:
        for s in range(steps):
            ctx.mc_step(P, fields, s, out, counters=cnt)
    ctx.sort_products(out)
    return [t.cpu() for t in (P.px, P.py, P.pz, P.tau, P.flags)], out.to_numpy(), sfq.counters_dict(cnt)


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
    for k in a[1]:
        assert np.array_equal(a[1][k].view(np.uint8), b[1][k].view(np.uint8)), k
    assert a[2] == b[2]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["soa", "wave"])
def test_step_shapes_on_mixed_populations(kind, precision):
    """Every block shape of the TMA-staged kernel, around its tiles, gives the bits of the
    warp-streaming kernel: two particles of a lane in every combination of species and dead."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=4)
    for n in (1, 2, 480, 511, 960, 961, 1023, 1025, 160 * 1024 + 33):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        beam = _mixed_population(n, ctx.dtype, n)
        if kind == "soa":
            F = sfq.FieldSource.soa(*[(100 * torch.randn(n, generator=g, device="cuda")).to(ctx.dtype) for _ in range(6)])
        else:
            k0 = torch.randint(0, W.K_TABLE + 3, (n,), generator=g, device="cuda", dtype=torch.int32)
            amp = None if n % 2 else (300 * torch.rand(n, generator=g, device="cuda")).to(ctx.dtype)
            F = sfq.FieldSource.plane_wave(k0, torch.as_tensor(W.cos_table(np.float64)).to("cuda", ctx.dtype), W.K_STEP,
                                           amp=amp, amp0=150.0)
        ctx.set_step_shape(1)
        want = _run_mixed(ctx, beam, F, 3)
        assert want[2]["emitted"] > 0 or n < 400
        for shape in (0, 8, 16, 20):
            ctx.set_step_shape(2, shape)
            _same(_run_mixed(ctx, beam, F, 3), want)
        if kind == "wave":
            _same(_run_mixed(ctx, beam, F, 3, fused=True), want)
