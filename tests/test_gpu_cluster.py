"""The cluster form of the chain (few positions, M = 128) does the arithmetic
of the one-block form: gradients, losses and far fields agree bit for bit with
launches that take the latter (multi-problem calls, and more positions than the
cluster form takes), and recompute mode with the oracle."""
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


def _geom(wl, n=None):
    from paper_2205_06327_gb300 import api
    return api.Geometry(wl.M, wl.S, wl.H, wl.W, wl.N if n is None else n, wl.lambda_A, wl.dz_A, wl.pixel_A)


def _tensors(wl, I, dev, n=None):
    return (to_dev(wl.pos[:n], torch.int32, dev), to_dev(wl.probe, torch.complex64, dev),
            to_dev(wl.obj, torch.complex64, dev), to_dev(I[:n], torch.float32, dev))


@pytest.mark.parametrize("S,ny,nx", [(1, 1, 1), (2, 1, 3), (5, 3, 7), (3, 6, 8), (3, 7, 7)])
def test_cluster_matches_one_block(dev, S, ny, nx):
    from paper_2205_06327_gb300 import api
    from paper_2205_06327_gb300.multi import MultiProblem, Problem
    wl = synth.workload_random(128, S, ny, nx, 5, seed=800 + S + nx, amp_jitter=0.1)
    I = np.abs(synth.rng(1).normal(size=(wl.N, 128, 128))).astype(np.float32)
    t = _tensors(wl, I, dev)
    plan = api.Plan(_geom(wl), dev)
    loss, gO, gP = plan.loss_grad(*t)
    only = plan.loss_grad(*t, want_obj=False, want_probe=False)[0]
    mp = MultiProblem([Problem(_geom(wl), *t)], dev)
    lm, grads = mp.loss_grad_all()
    torch.cuda.synchronize()
    assert torch.equal(loss, lm[0]) and torch.equal(only, loss)
    assert torch.equal(gO, grads[0][0]) and torch.equal(gP, grads[0][1])
    plan.close()
    mp.close()


@pytest.mark.parametrize("S,N", [(4, 160), (9, 170), (16, 304 + 20), (12, 456 + 9), (2, 160), (2, 152)])
def test_cluster_tail_beside_the_accumulation(dev, S, N):
    """A chunk whose chain ends in a few positions: whichever form they take, beside
    the accumulation of the full waves, the result is the multi-problem call's (one
    launch of one-block chains) bit for bit."""
    from paper_2205_06327_gb300 import api
    from paper_2205_06327_gb300.multi import MultiProblem, Problem
    wl = synth.workload_random(128, S, 1, 2, 5, seed=840 + S, amp_jitter=0.1)
    g = torch.Generator(device=dev).manual_seed(S)
    pos = torch.stack([torch.randint(0, wl.H - 127, (N,), device=dev, generator=g),
                       torch.randint(0, wl.W - 127, (N,), device=dev, generator=g)], 1).int()
    t = (pos, to_dev(wl.probe, torch.complex64, dev), to_dev(wl.obj, torch.complex64, dev),
         torch.rand(N, 128, 128, device=dev, generator=g))
    plan = api.Plan(_geom(wl, N), dev)
    loss, gO, gP = plan.loss_grad(*t)
    mp = MultiProblem([Problem(_geom(wl, N), *t)], dev)
    lm, grads = mp.loss_grad_all()
    torch.cuda.synchronize()
    assert torch.equal(loss, lm[0]) and torch.equal(gO, grads[0][0]) and torch.equal(gP, grads[0][1])
    plan.close()
    mp.close()


def test_cluster_forward_matches_one_block(dev):
    from paper_2205_06327_gb300 import api
    wl = synth.workload_random(128, 3, 8, 8, 4, seed=811, amp_jitter=0.1)
    I = np.zeros((wl.N, 128, 128), np.float32)
    pos, probe, obj, _ = _tensors(wl, I, dev)
    ref = api.Plan(_geom(wl), dev).forward(pos, probe, obj, want_intensity=True)
    few = api.Plan(_geom(wl, 11), dev).forward(pos[:11], probe, obj, want_intensity=True)
    torch.cuda.synchronize()
    assert torch.equal(ref[0][:11], few[0]) and torch.equal(ref[1][:11], few[1])


@pytest.mark.parametrize("S,L", [(4, 1), (5, 2), (7, 3)])
def test_cluster_recompute_and_window_outside(dev, S, L):
    from paper_2205_06327_gb300 import api
    from paper_2205_06327_gb300._lib import PtychoError
    wl = synth.workload_random(128, S, 1, 3, 9, seed=820 + S, amp_jitter=0.1)
    # At the true object the residual would be 1 - 1.1^-1/2 = 4.7 % of the
    # amplitude everywhere, so the loss would take the forward chain's relative
    # error 2 / 0.047 = 43 times: 1e-5 is out of reach there at 2.5e-7 (FP32 over
    # five slices).  The perturbed start has residuals of the amplitude's size.
    I = (measurements(wl) * 1.1).astype(np.float32)
    wl.obj = start_object(wl, "perturbed", S)
    keep = [0, 2]
    F, gO, gP = orc.loss_grad(c64(wl.probe), c64(wl.obj), wl.pos[keep], I[keep].astype(np.float64), propagator(wl))
    wl.pos[1] = (wl.H - 127, 0)
    plan = api.Plan(_geom(wl), dev, ckpt_every=L, async_check=True)
    l, go, gp = plan.loss_grad(*_tensors(wl, I, dev))
    torch.cuda.synchronize()
    with pytest.raises(PtychoError):
        plan.status()
    assert abs(l.item() - F) <= TOL_FP32 * F
    assert rel_l2(go.cpu().numpy(), gO) <= TOL_FP32 and rel_l2(gp.cpu().numpy(), gP) <= TOL_FP32
    plan.close()


@pytest.mark.parametrize("n,S,L", [(1, 2, 0), (3, 4, 0), (2, 5, 2)])
def test_cluster_wait_that_expires_is_reported(dev, n, S, L):
    """With PTYCHO_FLAG_SELFTEST_TIMEOUT the blocks of a cluster send nothing
    and wait for one another anyway: the short wait expires, the kernel ends (no
    further waits, however many exchanges follow), an asynchronous call leaves
    PTYCHO_ERR_TIMEOUT for ptycho_plan_status, calls that read a scalar on the
    host return it, a line search leaves the unknowns alone, and the next
    evaluation on the GPU is right."""
    import ctypes as C

    from paper_2205_06327_gb300 import _lib
    wl = synth.workload_random(128, S, 1, n, 9, seed=830 + S, amp_jitter=0.1)
    I = (measurements(wl) * 1.1).astype(np.float32)
    wl.obj = start_object(wl, "perturbed", S)
    pos, probe, obj, meas = _tensors(wl, I, dev)
    lib = _lib.load()
    p = _lib.PtychoParams(M=wl.M, S=wl.S, H=wl.H, W=wl.W, N=wl.N, lambda_A=wl.lambda_A, dz_A=wl.dz_A,
                          pixel_A=wl.pixel_A, ckpt_every=L, flags=_lib.PTYCHO_FLAG_SELFTEST_TIMEOUT)
    h = C.c_void_p()
    st = torch.cuda.current_stream(dev).cuda_stream
    assert lib.ptycho_plan_create(C.byref(h), C.byref(p)) == _lib.PTYCHO_OK
    gO, gP = torch.empty_like(obj), torch.empty_like(probe)
    loss = torch.zeros((), dtype=torch.float64, device=dev)
    args = (pos.data_ptr(), probe.data_ptr(), obj.data_ptr(), meas.data_ptr())
    assert lib.ptycho_loss_grad(h, *args, loss.data_ptr(), gO.data_ptr(), gP.data_ptr(), st) == _lib.PTYCHO_OK
    torch.cuda.synchronize()
    assert lib.ptycho_plan_status(h) == _lib.PTYCHO_ERR_TIMEOUT
    assert lib.ptycho_plan_status(h) == _lib.PTYCHO_OK  # reading clears it
    hl, t = C.c_double(0.0), C.c_double(0.0)
    for grads in ((gO.data_ptr(), gP.data_ptr()), (None, None)):
        assert lib.ptycho_loss_grad(h, *args, C.addressof(hl), *grads, st) == _lib.PTYCHO_ERR_TIMEOUT
        assert b"gave up" in lib.ptycho_last_error()
        assert lib.ptycho_plan_status(h) == _lib.PTYCHO_OK  # the call has reported and cleared it
    probe2, obj2 = probe.clone(), obj.clone()
    assert lib.ptycho_step(h, pos.data_ptr(), probe2.data_ptr(), obj2.data_ptr(), meas.data_ptr(), 0.1, 0.1, 1,
                           None, C.addressof(t), st) == _lib.PTYCHO_ERR_TIMEOUT
    torch.cuda.synchronize()
    assert torch.equal(probe2, probe) and torch.equal(obj2, obj)
    assert lib.ptycho_plan_destroy(h) == _lib.PTYCHO_OK
    if L == 0:
        assert lib.ptycho_loss_grad_noalloc(C.byref(p), *args, C.addressof(hl), gO.data_ptr(), gP.data_ptr(),
                                            st) == _lib.PTYCHO_ERR_TIMEOUT
    p.flags = 0
    assert lib.ptycho_plan_create(C.byref(h), C.byref(p)) == _lib.PTYCHO_OK
    assert lib.ptycho_loss_grad(h, *args, C.addressof(hl), gO.data_ptr(), gP.data_ptr(), st) == _lib.PTYCHO_OK
    assert lib.ptycho_plan_status(h) == _lib.PTYCHO_OK
    F, rO, rP = orc.loss_grad(c64(wl.probe), c64(wl.obj), wl.pos, I.astype(np.float64), propagator(wl))
    assert abs(hl.value - F) <= TOL_FP32 * F
    assert rel_l2(gO.cpu().numpy(), rO) <= TOL_FP32 and rel_l2(gP.cpu().numpy(), rP) <= TOL_FP32
    assert lib.ptycho_plan_destroy(h) == _lib.PTYCHO_OK
