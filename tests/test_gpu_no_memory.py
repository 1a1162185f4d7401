"""Calls that go on after one that found no room on the device: the status is
STAGGER_EOOM, nothing of it is left to the next call, and with room again the same
context gives the values it would have given."""
import pytest
import torch

import workloads as inputs

pytestmark = pytest.mark.gpu

N = 64
ARRAY = 4 * N ** 3          # one FP32 array
DT = 1e-3


def state():
    import paper_2405_02483_gb300 as S
    w = inputs.orszag_tang_3d(N)
    refs, dev = S.split_state(w.fields)
    p = S.default_params(ref=refs, nu1=0.04, nu2=1.0, nu3=0.04, nuE=1.0, nuB=1.0, do_quench=1)
    gen = torch.Generator(device="cuda").manual_seed(3)
    return p, dev, [torch.randn((N, N, N), generator=gen, device="cuda") for _ in range(8)]


def make(p):
    import paper_2405_02483_gb300 as S
    return S.Sim((N, N, N), (1.0 / N,) * 3, p)


def same(got, want):
    """Compared on the host: torch takes no device memory for it."""
    return all(torch.equal(a.cpu(), b.cpu()) for a, b in zip(got, want))


def hold(room):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")


# Arrays free before the adjoint: for part of the 181 node values; for them but no
# cotangents; for all but the workspace (the lean layout takes 292).  The same beside
# node values that a right-hand side has already taken.
@pytest.mark.parametrize("forward_first,room", [(False, 60), (False, 200), (False, 286), (True, 20),
                                                (True, 105)])
def test_calls_after_an_adjoint_without_room(forward_first, room):
    import paper_2405_02483_gb300 as S
    p, dev, lam = state()
    ref = make(p)
    want_f, want_u = ref.rhs(dev), ref.rhs_unfused(dev)
    want_a = ref.step_adjoint(dev, DT, lam)
    ref.close()
    sim = make(p)
    out, got = [torch.empty_like(t) for t in lam], [torch.empty_like(t) for t in lam]
    if forward_first:
        sim.rhs_unfused(dev, out=got)
    held = hold(room * ARRAY)
    try:
        with pytest.raises(S.StaggerError) as e:
            sim.step_adjoint(dev, DT, lam, out=out)
        assert e.value.status == S.EOOM
        sim.rhs(dev, out=got)
        assert same(got, want_f)
        if room == 60:   # (nothing of the graph fits)
            with pytest.raises(S.StaggerError) as e:
                sim.rhs_unfused(dev, out=got)
            assert e.value.status == S.EOOM
        else:
            sim.rhs_unfused(dev, out=got)
            assert same(got, want_u)
        if room < 100:   # (a context takes about 90)
            with pytest.raises(S.StaggerError) as e:
                make(p)
            assert e.value.status == S.EOOM
            sim.rhs(dev, out=got)
    finally:
        del held
        torch.cuda.empty_cache()
    sim.rhs_unfused(dev, out=got)
    assert same(got, want_u)
    sim.step_adjoint(dev, DT, lam, out=out)
    assert same(out, want_a)
    sim.close()
