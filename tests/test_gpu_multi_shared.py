"""Multi-problem calls whose problems share memory that one of them writes: the
generic windows' problems run first, then the register-resident ones, so the
results are those of the single calls in that order, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _problems(dev, windows, S=3, H=190, W=201, ny=4, nx=5):
    from paper_2205_06327_gb300 import api
    from paper_2205_06327_gb300.multi import Problem
    out = []
    for k, M in enumerate(windows):
        g = torch.Generator(device=dev).manual_seed(70 + k)
        pos = torch.tensor([[9 * (i // nx), 7 * (i % nx)] for i in range(ny * nx)], dtype=torch.int32, device=dev)
        probe = torch.randn(M, M, dtype=torch.complex64, device=dev, generator=g) / M
        obj = torch.exp(0.3j * torch.rand(S, H, W, device=dev, generator=g))
        meas = torch.rand(ny * nx, M, M, device=dev, generator=g) / M
        out.append(Problem(api.Geometry(M, S, H, W, ny * nx), pos, probe, obj, meas))
    return out


@pytest.mark.parametrize("writer", ["generic", "register-resident"])
@pytest.mark.parametrize("shift", [0, 1])  # the whole array, or an overlap by all but its first slice
def test_gradient_of_one_problem_lands_in_the_object_of_another(dev, writer, shift):
    from paper_2205_06327_gb300 import _lib
    from paper_2205_06327_gb300.api import _stream_handle
    from paper_2205_06327_gb300.multi import MultiProblem
    probs = _problems(dev, [64, 96, 128, 108])
    src, dst = (1, 2) if writer == "generic" else (0, 3)
    S, H, W = probs[dst].obj.shape
    both = torch.empty(2 * S, H, W, dtype=torch.complex64, device=dev)
    grad, shared = both[:S], both[shift:shift + S]  # the writer's gradient, the reader's object
    start = probs[dst].obj
    probs[dst].obj = shared
    grads = [(grad if k == src else torch.empty_like(start), torch.empty_like(p.probe)) for k, p in enumerate(probs)]
    mp = MultiProblem(probs, dev)

    def reset():
        both.zero_()
        shared.copy_(start)
        for k, (gO, gP) in enumerate(grads):
            gP.fill_(5)
            if k != src:
                gO.fill_(5)

    reset()
    for k in (1, 3, 0, 2):
        p = probs[k]
        mp.plans[k].loss_grad(p.pos, p.probe, p.obj, p.meas, out_obj=grads[k][0], out_probe=grads[k][1])
    torch.cuda.synchronize()
    want = [both.clone()] + [t.clone() for g in grads for t in g]
    reset()
    torch.cuda.synchronize()
    arr = mp._entries(grads)
    with torch.cuda.device(dev):
        _lib.check(mp.plans[0].lib.ptycho_multi_loss_grad(arr, len(probs), _stream_handle(dev)))
    torch.cuda.synchronize()
    mp.check_status()
    assert all(torch.equal(a, b) for a, b in zip(want, [both] + [t for g in grads for t in g]))
    mp.close()
