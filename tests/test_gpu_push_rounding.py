"""The binary64 push's arithmetic: its factors' bits, and where their argument overflows."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2301_07684_gb300 import sfq
from paper_2301_07684_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _push(px, pz, bz, dt, precision="fp64"):
    """Positrons of momentum (px, 0, pz) pushed in the field (0, 0, bz) alone."""
    n = len(px)
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision=precision, seed=1)
    dev = lambda a: torch.as_tensor(np.broadcast_to(np.asarray(a, np.float64), (n,)).copy()).to("cuda", ctx.dtype)
    flags = torch.full((n,), sfq.SFQ_ALIVE | (sfq.SFQ_POSITRON << sfq.SFQ_SPECIES_SHIFT), dtype=torch.uint8, device="cuda")
    P = sfq.ParticleBuffers(dev(px), dev(0.0), dev(pz), torch.ones(n, dtype=torch.float64, device="cuda"), flags)
    ctx.push(P, sfq.FieldSource.soa(dev(0.0), dev(0.0), dev(0.0), dev(0.0), dev(0.0), dev(bz)), 0, dt)
    got = [t.double().cpu().numpy() for t in (P.px, P.py, P.pz)]
    ctx.close()
    return got


def test_rotation_by_a_field_whose_square_overflows():
    """t = h B / gamma, s = 2 t / (1 + t.t): with 1 + t.t infinite, s is zero and the momentum
    stays; just below, the momentum turns by pi (to 2 / t, below 1e-150).  Tolerance: ten
    roundings of terms of at most 2 |u| (the products u' s and their factors), 20 * 2^-53."""
    px = np.array([1.0, 3.0, 1234.5, 2.0, 700.0, 1.0])
    t = np.array([1e160, 1e200, 1e300, 1.3e154, 1.2e154, 1e152])        # the last three squares are finite
    gamma = np.sqrt(1 + px * px + 0.25)
    x, y, z = _push(px, 0.5, t * gamma, 2.0)                            # h = dt / 2 = 1
    want = np.where(t >= 1e160, px, -px)
    assert np.abs(x / want - 1).max() < 20 * 2.0 ** -53, x
    assert np.abs(y / px).max() < 20 * 2.0 ** -53, y
    assert np.array_equal(z, np.full(6, 0.5))


def test_factors_are_rounded_as_the_formula_says():
    """With u = (1, 0, pz) and B along z, u_y = -s = -2 t / (1 + t^2), t = h B / gamma: every
    operation of it is correctly rounded (root, divisions, products, 1 + t^2 with one
    rounding), so the result has the bits of the same operations on the host."""
    g = np.random.default_rng(3)
    n = 20000
    pz, bz = 10.0 ** g.uniform(-2, 5, n), 10.0 ** g.uniform(-2, 6, n)
    pz[: n // 2] = 0.0                                     # gamma^2 = 2
    _, y, _ = _push(np.ones(n), pz, bz, 2.0)
    one_plus_square = np.array([float(1 + Fraction(v) ** 2) for v in pz.tolist()])
    g2 = np.array([float(1 + Fraction(v)) for v in one_plus_square.tolist()])
    t = (1.0 / np.sqrt(g2)) * bz
    d = np.array([float(1 + Fraction(v) ** 2) for v in t.tolist()])
    assert np.array_equal(y, -((2.0 / d) * t))
