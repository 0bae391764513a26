"""The object-gradient accumulation's bands at the sizes where they can go
wrong: odd windows (8-byte loads), windows wider than a warp's loads in flight,
objects of one row band and of several column tiles, rows that no window or
every window covers, more positions than one list, and tiles asked for."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from paper_2205_06327_gb300 import synth
from tests.helpers import TOL_FP32, c64, measurements, propagator, rel_l2, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _grad(wl, I, dev, pos=None, **kw):
    from paper_2205_06327_gb300 import api
    pos = wl.pos if pos is None else pos
    plan = api.Plan(api.Geometry(wl.M, wl.S, wl.H, wl.W, len(pos), wl.lambda_A, wl.dz_A, wl.pixel_A), dev, **kw)
    out = plan.loss_grad(to_dev(pos, torch.int32, dev), to_dev(wl.probe, torch.complex64, dev),
                         to_dev(wl.obj, torch.complex64, dev), to_dev(I, torch.float32, dev))
    torch.cuda.synchronize()
    plan.close()
    return out[1].cpu().numpy()


@pytest.mark.parametrize("M,S,ny,nx,step,H,W", [
    (9, 2, 3, 5, 4, None, None), (16, 2, 4, 9, 5, None, None), (27, 1, 1, 3, 11, 27, 700),
    (64, 2, 2, 3, 9, 64, 90), (64, 1, 2, 3, 9, 200, 1500), (96, 1, 3, 3, 7, 101, 131), (648, 1, 1, 2, 5, None, None)])
def test_bands_match_oracle(dev, M, S, ny, nx, step, H, W):
    wl = synth.workload_random(M, S, ny, nx, step, seed=500 + M + S, amp_jitter=0.1)
    if H is not None:  # the same scan on another object extent, spread over its width
        g = synth.rng(600 + M)
        wl.H, wl.W = H, W
        wl.obj = np.exp(0.3j * g.uniform(0, 1, size=(S, H, W))) * (1 + 0.1 * g.uniform(-1, 1, size=(S, H, W)))
        wl.pos = np.stack([g.integers(0, H - M + 1, wl.N), g.integers(0, W - M + 1, wl.N)], 1).astype(np.int32)
    I = (measurements(wl) * 1.2).astype(np.float32)
    gO = orc.loss_grad(c64(wl.probe), c64(wl.obj), wl.pos, I.astype(np.float64), propagator(wl))[1]
    ref = _grad(wl, I, dev)
    assert rel_l2(ref, gO) <= TOL_FP32
    for tile in ((8, 8), (32, 32), (4, 300), (1, 8000)):
        assert np.array_equal(ref, _grad(wl, I, dev, tile=tile))


def test_bands_more_positions_than_a_list(dev):
    """2600 positions (three lists): the gradient agrees with the oracle, and with
    the sum of two halves to reassociation."""
    wl = synth.workload_random(16, 1, 52, 50, 1, seed=777, amp_jitter=0.1)
    I = (measurements(wl) * 1.2).astype(np.float32)
    gO = orc.loss_grad(c64(wl.probe), c64(wl.obj), wl.pos, I.astype(np.float64), propagator(wl))[1]
    g = _grad(wl, I, dev)
    assert rel_l2(g, gO) <= TOL_FP32
    h = wl.N // 2
    halves = _grad(wl, I[:h], dev, pos=wl.pos[:h]) + _grad(wl, I[h:], dev, pos=wl.pos[h:])
    assert rel_l2(g, halves) <= 1e-6
