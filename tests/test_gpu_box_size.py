"""The derivative of a periodic field does not depend on how many of its periods
the box holds: a field and its repetition, which runs the kernels and thread-block
shapes of larger boxes, have the same right-hand side bit for bit, and ten quenched
Courant steps of a plane and of its repetition the same states (the quench, whose
ratio is steep where a stress is small, makes 1e-4 to 2e-3 of the rms in a cell of a
last bit)."""
import numpy as np
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu

RM = dict(nu1=0.04, nu2=1.0, nu3=0.04, nuE=1.0, nuB=1.0)


def fields(shape, seed):
    flat = shape[2] == 1
    u = inputs.solenoidal_velocity(shape, seed, 0.4, kmax=8.0, solenoidal=False)
    b = inputs.solenoidal_velocity(shape, seed + 1, 0.3, kmax=8.0)
    w = inputs.solenoidal_velocity(shape, seed + 2, 0.2, kmax=8.0, solenoidal=False)
    zero = np.zeros_like(u[0])
    noise = np.random.default_rng(seed).standard_normal((4,) + u[0].shape)   # rough from cell to cell
    u = [c + 0.02 * n for c, n in zip(u, noise)]
    b = [b[0] + 0.02 * noise[3], b[1], b[2]]
    return [1 + w[0], u[0], u[1], zero if flat else u[2], 0.9 + w[1], b[0], b[1],
            zero if flat else 0.3 + b[2]]


def tiled(dev, times):
    return [t.repeat(times[2], times[1], times[0]).contiguous() for t in dev]


@pytest.mark.parametrize("kw", [dict(), RM, dict(RM, do_quench=1), dict(RM, csmag=0.1, do_quench=1)])
@pytest.mark.parametrize("shape,times", [((64, 64, 64), (2, 2, 2)), ((64, 48, 44), (1, 3, 3)),
                                         ((32, 72, 52), (1, 3, 4)), ((44, 52, 36), (3, 3, 3))])
def test_rhs_of_a_repeated_field(shape, times, kw):
    import paper_2405_02483_gb300 as S
    refs, dev = S.split_state(fields(shape, 11), [1.0, 0, 0, 0, 0.9, 0, 0, 0.3])
    out = []
    for t in ((1, 1, 1), times):
        big = tuple(n * m for n, m in zip(shape, t))
        sim = S.Sim(big, (1.0 / 64,) * 3, S.default_params(ref=refs, **kw))
        out.append([a.clone() for a in sim.rhs(tiled(dev, t))])
        sim.close()
    for a, e in zip(out[1], tiled(out[0], times)):
        assert torch.equal(a, e)


@pytest.mark.parametrize("kw", [dict(), RM, dict(RM, do_quench=1), dict(RM, do_quench=1, quench_max3=1),
                                dict(RM, csmag=0.1, c1=-0.3, do_quench=1, do_2nddiv=1, d2lnr_lim=0.05),
                                dict(nu_const=1e-3), dict(RM, g=(0.1, 0.0, -0.2), t_cool=0.3, e_cool=0.8,
                                                          cor_L0=0.5, cor_Tunit=8e3)])
@pytest.mark.parametrize("shape,times", [((65, 40, 36), (1, 2, 2)), ((131, 38, 30), (1, 2, 3)),
                                         ((43, 52, 36), (3, 2, 2)), ((350, 250, 1), (3, 1, 1))])
def test_rhs_of_a_repeated_field_on_padded_rows(shape, times, kw):
    """One-cell threads on the small box's rows, padded rows on the large one's."""
    test_rhs_of_a_repeated_field(shape, times, kw)


def test_steps_of_a_repeated_plane():
    import paper_2405_02483_gb300 as S
    shape, times = (512, 512, 1), (2, 2, 1)
    refs, dev = S.split_state(fields(shape, 21), [1.0, 0, 0, 0, 0.9, 0, 0, 0])
    out = []
    for t in ((1, 1, 1), times):
        f = tiled(dev, t)
        sim = S.Sim((shape[0] * t[0], shape[1] * t[1], 1), (1.0 / 512,) * 3,
                    S.default_params(ref=refs, do_quench=1, **RM))
        sim.run(f, 10)
        out.append(f)
        sim.close()
    for a, e in zip(out[1], tiled(out[0], times)):
        assert torch.equal(a, e)
