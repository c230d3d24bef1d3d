"""The autotuner's shapes: what it times and returns is a fixed launch shape, which the context
takes as its own."""
import numpy as np
import pytest
import torch

from paper_2301_07684_gb300 import sfq
from paper_2301_07684_gb300 import workloads as W
from test_gpu_launch_rules import _mixed_population, _run_mixed, _same

pytestmark = pytest.mark.gpu


def _fields(kind, n, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if kind == "soa":
        return sfq.FieldSource.soa(*[(100 * torch.randn(n, generator=g, device="cuda")).to(dtype) for _ in range(6)])
    k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device="cuda", dtype=torch.int32)
    return sfq.FieldSource.plane_wave(k0, torch.as_tensor(W.cos_table(np.float64)).to("cuda", dtype), W.K_STEP, amp0=150.0)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["soa", "wave"])
def test_the_shape_of_15_warps_can_be_named(kind, precision):
    """15 warps with the plane wave; fields in memory take their default shape.  The bits are
    the warp-streaming kernel's."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=4)
    n = 20 * 1024 + 33
    beam, F = _mixed_population(n, ctx.dtype, n), _fields(kind, n, ctx.dtype, n)
    ctx.set_step_shape(1)
    want = _run_mixed(ctx, beam, F, 2)
    for grid in (0, 3):
        ctx.set_step_shape(2, 15, grid)
        _same(_run_mixed(ctx, beam, F, 2), want)
    for variant, shape in ((2, 14), (2, 17), (2, 19), (2, 4), (1, 15), (0, 15)):
        with pytest.raises(sfq.SfqError):
            ctx.set_step_shape(variant, shape)


@pytest.mark.parametrize("truncated", [False, True])
@pytest.mark.parametrize("kind", ["soa", "wave"])
def test_autotuned_shape_is_a_fixed_one(kind, truncated):
    """The shape returned is a number of particles per lane or warps per block, never "default":
    it is what the sample was timed with, and the whole population runs it."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    if truncated:
        ctx.set_sampler_coefficients(8)
    n = 1 << 22
    beam = _mixed_population(n, ctx.dtype, n)
    F = _fields(kind, n, ctx.dtype, n)
    P = sfq.ParticleBuffers(*[t.clone() for t in beam])
    for sample in (0, 1 << 20):
        variant, shape, ms = ctx.autotune_step(P, F, 0, sample_n=sample)
        assert ms > 0.0
        assert shape in ({1: (2,), 2: (16,)} if truncated else
                         {1: (1, 2, 4), 2: (8, 15, 16, 20) if kind == "wave" else (8, 16, 20)})[variant]
        ctx.set_step_shape(variant, shape)
