"""The FP64 adjoint where the device has no room for the node values of all three
stages: with one set each stage is evaluated again in the reverse, and the gradient is
the same bit for bit.  Room for all but the cotangents (the graph itself takes the lean
layout) and for all but the workspace (it is rebuilt)."""
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("room", [600, 660])   # arrays; three sets, scratch, cotangents, workspace: 692
def test_fp64_adjoint_with_one_set_of_values(room):
    import paper_2405_02483_gb300 as S
    n = 64
    array = 8 * n ** 3
    w = inputs.orszag_tang_3d(n)
    refs, dev = S.split_state(w.fields)
    p = S.default_params(ref=refs, nu1=0.04, nu2=1.0, nu3=0.04, nuE=1.0, nuB=1.0, do_quench=1)
    f = [t.double() for t in dev]
    gen = torch.Generator(device="cuda").manual_seed(3)
    lam = [torch.randn((n, n, n), generator=gen, device="cuda", dtype=torch.float64) for _ in range(8)]
    out = [torch.empty_like(t) for t in lam]

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    def adjoint(room=None):
        sim = S.Sim((n, n, n), (1.0 / n,) * 3, p)
        hold = torch.empty(free() - room * array, dtype=torch.uint8, device="cuda") if room else None
        before = free()
        try:
            sim.step_adjoint_f64(f, 1e-3, lam, out=out)
            took = before - free()
        finally:
            del hold
            torch.cuda.empty_cache()
            sim.close()
        return [t.clone() for t in out], took / array

    adjoint()                      # loads the kernels
    ref, full = adjoint()
    got, lean = adjoint(room)
    assert full > 680 and lean < 310
    for a, e in zip(got, ref):
        assert torch.equal(a, e)
