"""The TMA-staged step's ring of stages, many times round: a small grid gives a block dozens of
tiles, so every stage is filled, handed over and released again and again."""
import pytest
import torch

from paper_2301_07684_gb300 import sfq
from paper_2301_07684_gb300 import workloads as W
from test_gpu_launch_rules import _mixed_population, _run_mixed, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["soa", "wave"])
def test_stages_are_reused(kind, precision):
    """Every block shape on two and three blocks gives the bits of the warp-streaming kernel."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=4)
    n = 160 * 1024 + 33
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    beam = _mixed_population(n, ctx.dtype, n)
    if kind == "soa":
        F = sfq.FieldSource.soa(*[(100 * torch.randn(n, generator=g, device="cuda")).to(ctx.dtype) for _ in range(6)])
    else:
        k0 = torch.randint(0, W.K_TABLE, (n,), generator=g, device="cuda", dtype=torch.int32)
        amp = (300 * torch.rand(n, generator=g, device="cuda")).to(ctx.dtype)
        F = sfq.FieldSource.plane_wave(k0, torch.as_tensor(W.cos_table()).to("cuda", ctx.dtype), W.K_STEP, amp=amp)
    ctx.set_step_shape(1)
    want = _run_mixed(ctx, beam, F, 2)
    assert want[2]["emitted"] > 0 and want[2]["timeouts"] == 0
    for shape in (0, 8, 16, 20):
        for grid in (2, 3):
            ctx.set_step_shape(2, shape, grid)
            _same(_run_mixed(ctx, beam, F, 2), want)
