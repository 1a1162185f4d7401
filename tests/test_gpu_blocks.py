"""Shapes on which the fused kernels' block rules take another branch, at the
edges of their tiles: 32, 16 and 8 lanes along x (rows that do not fill a whole
block, tiles that hang over the box in x and y), with the edge heating densities
centred through shared memory; and rows of no multiple of four cells, which run on
padded copies with periodic images (the shortest row, each remainder, one plane).

Four-cell against one-cell threads: the same FP32 operations but for contraction
and the order of the two centring passes.  Tolerance 2e-5 of the term scale, that
of the mapping test on small boxes."""
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu


RM = dict(nu1=0.04, nu2=1.0, nu3=0.04)
# every derivative of the stress two-point (a negative limit flags all cells)
OPTS = dict(RM, csmag=0.1, c1=-0.3, do_2nddiv=1, d2lnr_lim=-1.0, g=(0.1, 0.0, -0.2), t_cool=0.3,
            e_cool=0.8, cor_L0=0.5, cor_Tunit=8e3)


@pytest.mark.parametrize("shape,kw", [
    ((128, 53, 156), RM), ((64, 75, 220), RM), ((160, 60, 110), RM), ((1024, 1028, 1), RM),
    ((132, 51, 160), RM), ((128, 3, 2800), RM),
    ((131, 97, 75), RM), ((61, 60, 61), RM), ((62, 61, 59), {}), ((63, 1, 3300), OPTS),
    ((9, 150, 150), OPTS), ((1021, 200, 1), RM), ((127, 65, 29), dict(nu_const=1e-3)), ((66, 57, 60), OPTS)])
def test_four_cell_blocks_match_one_cell(shape, kw):
    import paper_2405_02483_gb300 as S
    nx, ny, nz = shape
    u = inputs.solenoidal_velocity(shape, 5, 0.3, kmax=3.0, solenoidal=False)
    b = inputs.solenoidal_velocity(shape, 6, 0.2, kmax=3.0)
    f = [1 + 0.1 * u[0], u[0], u[1], u[2], 0.9 + 0.1 * u[1], b[0], b[1], 0.3 + b[2]]
    out = []
    for scalar in (0, 1):
        refs, dev = S.split_state(f, [1.0, 0, 0, 0, 0.9, 0, 0, 0.3])
        sim = S.Sim(shape, tuple(1.0 / max(n, 8) for n in shape),
                    S.default_params(ref=refs, scalar_cells=scalar, **kw))
        rhs = [t.clone() for t in sim.rhs(dev)]
        sim.step(dev, 1e-4)
        dt = sim.step(dev, want_dt=True)
        out.append((rhs, dev, dt))
        sim.close()
    (r4, s4, d4), (r1, s1, d1) = out
    top = max(float(t.abs().max()) for t in r1)
    for a, e in zip(r4, r1):
        assert float((a - e).abs().max()) <= 2e-5 * max(float(e.abs().max()), 1e-3 * top)
    assert abs(d4 - d1) <= 1e-5 * d1
    for a, e in zip(s4, s1):
        assert float((a - e).abs().max()) <= 2e-5 * max(float(e.abs().max()), 1.0)
