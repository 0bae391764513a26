"""A host-checked call with a window outside the object: it is refused with
PTYCHO_ERR_POSITION, leaves every array of the caller as it was, and returns
with nothing of its own still running on them."""
import numpy as np
import pytest

from paper_2205_06327_gb300 import synth
from tests.helpers import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


@pytest.mark.parametrize("M,S,N,L", [(128, 16, 300, 0), (128, 16, 8, 0), (64, 24, 900, 0), (192, 10, 120, 0),
                                     (36, 6, 900, 0), (128, 12, 300, 4)])
def test_refused_call_leaves_arrays_and_stream_idle(dev, M, S, N, L):
    from paper_2205_06327_gb300 import api
    from paper_2205_06327_gb300._lib import PTYCHO_ERR_POSITION, PtychoError
    g = torch.Generator(device=dev).manual_seed(M + S)
    H, W = M + 40, M + 60
    pos = np.stack([synth.rng(1).integers(0, 41, N), synth.rng(2).integers(0, 61, N)], 1).astype(np.int32)
    pos[-1] = (41, 0)
    pos = to_dev(pos, torch.int32, dev)
    probe = torch.randn(M, M, dtype=torch.complex64, device=dev, generator=g) / M
    obj = torch.exp(0.3j * torch.rand(S, H, W, device=dev, generator=g))
    meas = torch.rand(N, M, M, device=dev, generator=g) / M
    plan = api.Plan(api.Geometry(M, S, H, W, N), dev, ckpt_every=L)
    gO, gP = torch.full_like(obj, 7.0), torch.full_like(probe, 7.0)
    probe2, obj2 = probe.clone(), obj.clone()
    for call in (lambda: plan.loss_grad(pos, probe, obj, meas, out_obj=gO, out_probe=gP),
                 lambda: plan.loss_grad(pos, probe, obj, meas, want_obj=False, want_probe=False),
                 lambda: plan.step(pos, probe2, obj2, meas, 0.1, 0.1),
                 lambda: plan.step(pos, probe2, obj2, meas, 0.1, 0.1, line_search=True)):
        torch.cuda.synchronize()
        with pytest.raises(PtychoError) as e:
            call()
        assert torch.cuda.current_stream(dev).query()
        assert e.value.code == PTYCHO_ERR_POSITION
    assert bool((gO == 7.0).all()) and bool((gP == 7.0).all())
    assert torch.equal(probe2, probe) and torch.equal(obj2, obj)
    plan.status()  # nothing left over for a later reader
    pos[-1, 0] = 40
    loss, gO, gP = plan.loss_grad(pos, probe, obj, meas)
    assert bool(torch.isfinite(loss)) and bool(torch.isfinite(torch.view_as_real(gO)).all())
    plan.close()
