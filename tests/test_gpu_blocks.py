"""Shapes on which the fused kernels' block rules take another branch, at the
edges of their tiles: 32, 16 and 8 lanes along x (rows that do not fill a whole
block, tiles that hang over the box in x and y), with the edge heating densities
centred through shared memory.

Four-cell against one-cell threads: the same FP32 operations but for contraction
and the order of the two centring passes.  Tolerance 2e-5 of the term scale, that
of the mapping test on small boxes."""
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(128, 53, 48), (64, 75, 66), (160, 60, 40), (1024, 308, 1),
                                   (132, 51, 50), (128, 3, 850)])
def test_four_cell_blocks_match_one_cell(shape):
    import paper_2405_02483_gb300 as S
    nx, ny, nz = shape
    u = inputs.solenoidal_velocity(shape, 5, 0.3, kmax=3.0, solenoidal=False)
    b = inputs.solenoidal_velocity(shape, 6, 0.2, kmax=3.0)
    f = [1 + 0.1 * u[0], u[0], u[1], u[2], 0.9 + 0.1 * u[1], b[0], b[1], 0.3 + b[2]]
    out = []
    for scalar in (0, 1):
        refs, dev = S.split_state(f, [1.0, 0, 0, 0, 0.9, 0, 0, 0.3])
        sim = S.Sim(shape, tuple(1.0 / max(n, 8) for n in shape),
                    S.default_params(ref=refs, nu1=0.04, nu2=1.0, nu3=0.04, scalar_cells=scalar))
        rhs = [t.clone() for t in sim.rhs(dev)]
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
