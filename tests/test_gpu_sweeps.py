"""The op graph's batched sweeps on shapes where the launch can go wrong: rows
that fill part of a block, one chunk of four cells (both neighbours wrap onto
it), one plane, no multiple of four, more than one block of lanes.

FP32 (four-cell threads where nx % 4 == 0) against the FP64 sweep (one-cell
threads) of the same step, constant viscosity, so that no switch separates the
two.  Tolerance, relative to the norm of the gradient: a cotangent sums about
300 terms, each rounded to 2^-24 with stencil weights of sum 2.5 in magnitude:
300 * 2.5 * 2^-24 = 4.5e-5."""
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 9, 5), (36, 8, 1), (132, 6, 7), (13, 8, 6), (64, 1, 33)])
def test_fp32_sweeps_match_fp64(shape):
    import paper_2405_02483_gb300 as S
    nx, ny, nz = shape
    u = inputs.solenoidal_velocity(shape, 5, 0.3, kmax=float(max(1, min(3, nx // 2))), solenoidal=False)
    b = inputs.solenoidal_velocity(shape, 6, 0.2, kmax=float(max(1, min(3, nx // 2))))
    f = [1 + 0.1 * u[0], u[0], u[1], u[2], 0.9 + 0.1 * u[1], b[0], b[1], 0.3 + b[2]]
    refs, dev = S.split_state(f, [1.0, 0, 0, 0, 0.9, 0, 0, 0.3])
    sp = tuple(1.0 / max(n, 8) for n in shape)
    sim = S.Sim(shape, sp, S.default_params(ref=refs, nu_const=1e-3, g=(0.1, 0.0, -0.2)))
    gen = torch.Generator(device="cuda").manual_seed(1)
    lam = [torch.randn((nz, ny, nx), generator=gen, device="cuda") for _ in range(8)]
    dt = 0.1 * min(sp)
    got = sim.step_adjoint(dev, dt, lam)
    ref = sim.step_adjoint_f64([t.double() for t in dev], dt, [t.double() for t in lam])
    for a, e in zip(got, ref):
        assert torch.isfinite(a).all()
        assert float((a.double() - e).norm() / e.norm()) <= 4.5e-5
    rhs = sim.rhs_unfused(dev)
    rhs64 = sim.rhs_unfused_f64([t.double() for t in dev])
    scale = max(float(e.norm()) for e in rhs64)
    for a, e in zip(rhs, rhs64):
        assert float((a.double() - e).norm()) <= 4.5e-5 * scale
