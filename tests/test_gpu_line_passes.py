"""GPU parity of the generic windows' line passes at the sizes where their
compile-time instances can go wrong: odd and even radix pairs, blocks whose
items do not fill the threads, two and three factors, one to four slices (each
first and last pass has its own form), recompute segments of one slice and
more, and a window outside the object next to windows inside."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from paper_2205_06327_gb300 import synth
from tests.helpers import TOL_FP32, c64, measurements, propagator, rel_l2, start_object, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _run(wl, obj, I, dev, pos=None, **kw):
    from paper_2205_06327_gb300 import api
    plan = api.Plan(api.Geometry(wl.M, wl.S, wl.H, wl.W, wl.N, wl.lambda_A, wl.dz_A, wl.pixel_A), dev, **kw)
    out = plan.loss_grad(to_dev(wl.pos if pos is None else pos, torch.int32, dev),
                         to_dev(wl.probe, torch.complex64, dev), to_dev(obj, torch.complex64, dev),
                         to_dev(I, torch.float32, dev))
    torch.cuda.synchronize()
    out = [t.cpu().numpy() for t in out]
    return out, plan


@pytest.mark.parametrize("M", [48, 72, 81, 96, 108, 144, 192, 256, 384, 512])
@pytest.mark.parametrize("S,L", [(1, 0), (2, 0), (4, 0), (4, 1), (5, 3)])
def test_line_pass_instances(dev, M, S, L):
    if M > 300 and S > 4:
        pytest.skip("covered by the smaller windows; the oracle takes long here")
    wl = synth.workload_random(M, S, 1, 2, 7, seed=300 + M + S, amp_jitter=0.1)
    I = (measurements(wl) * 1.15).astype(np.float32)
    obj = start_object(wl, "perturbed", S)
    F, gO, gP = orc.loss_grad(c64(wl.probe), c64(obj), wl.pos, I.astype(np.float64), propagator(wl))
    (l, go, gp), plan = _run(wl, obj, I, dev, ckpt_every=L)
    plan.status()
    assert abs(l - F) <= TOL_FP32 * F and rel_l2(go, gO) <= TOL_FP32 and rel_l2(gp, gP) <= TOL_FP32


@pytest.mark.parametrize("M", [81, 96, 384, 18])  # 18: the runtime radix schedule
def test_line_pass_window_outside_contributes_nothing(dev, M):
    from paper_2205_06327_gb300._lib import PtychoError
    wl = synth.workload_random(M, 3, 1, 3, 5, seed=400 + M, amp_jitter=0.1)
    I = (measurements(wl) * 1.1).astype(np.float32)
    keep = [0, 2]
    F, gO, gP = orc.loss_grad(c64(wl.probe), c64(wl.obj), wl.pos[keep], I[keep].astype(np.float64), propagator(wl))
    pos = wl.pos.copy()
    pos[1] = (0, wl.W - M + 1)
    (l, go, gp), plan = _run(wl, wl.obj, I, dev, pos=pos, async_check=True)
    with pytest.raises(PtychoError):
        plan.status()
    assert abs(l - F) <= TOL_FP32 * F and rel_l2(go, gO) <= TOL_FP32 and rel_l2(gp, gP) <= TOL_FP32


@pytest.mark.parametrize("M,W", [(1024, 2100000), (1152, 1880000)])  # an instance, the runtime radix schedule
def test_line_pass_window_of_a_very_wide_object(dev, M, W):
    """A window of an object so wide that its last rows lie 2^31 pixels and more
    from its first: the same window alone gives the same result bit for bit."""
    from paper_2205_06327_gb300 import api
    g = torch.Generator(device=dev).manual_seed(M)
    win = torch.exp(0.3j * torch.rand(1, M, M, device=dev, generator=g))
    meas = torch.rand(1, M, M, device=dev, generator=g) / M
    probe = to_dev(synth.defocused_probe(M, 0.15, np.pi * 0.15 * M, 1.0, energy=float(M)), torch.complex64, dev)
    wide = torch.ones(1, M, W, dtype=torch.complex64, device=dev)
    wide[:, :, W - M:] = win
    out = []
    for obj, x, width in ((win, 0, M), (wide, W - M, W)):
        plan = api.Plan(api.Geometry(M, 1, M, width, 1), dev)
        loss, gO, gP = plan.loss_grad(torch.tensor([[0, x]], dtype=torch.int32, device=dev), probe, obj, meas)
        out.append((loss, gO[:, :, x:x + M].clone(), gP))
        assert x == 0 or not torch.count_nonzero(gO[:, :, :x])
        plan.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
