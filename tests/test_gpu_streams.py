"""Contexts on streams of their own: the shape follows what else is in flight, the results do not."""

from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402
import phantoms  # noqa: E402

pytestmark = pytest.mark.gpu
STEP = 1.0 / np.sqrt(4.0 / 9.0 + 8.0)


def problem(H, S, seed):
    pb = phantoms.volume(H, H, S, seed=seed, lam=5e-4, n_iter=40)
    return torch.from_numpy(pb.field.copy()).cuda(), torch.from_numpy(pb.mask.copy()).cuda()


class Call:
    def __init__(self, H, S, seed, n_iter, stream, **opts):
        self.f, self.m = problem(H, S, seed)
        self.chi = torch.full_like(self.f, float("nan"))
        self.n_iter, self.stream = n_iter, stream
        torch.cuda.synchronize()
        self.ctx = pcs.pcs_create(H, H, S, stream=stream, **opts)

    def run(self):
        pcs.pcs_solve_slices(self.ctx, self.f, self.m, 5e-4, STEP, STEP, self.n_iter, self.chi)
        return pcs.pcs_last_variant(self.ctx)["cluster_size"]

    def close(self):
        pcs.pcs_check(self.ctx)
        pcs.pcs_destroy(self.ctx)
        return self.chi.cpu().numpy()


def test_one_slice_beside_a_volume_takes_a_small_cluster():
    """Tensor-memory clusters of two solves on two streams; same bits as alone."""
    st = [torch.cuda.Stream() for _ in range(2)]
    one = Call(256, 1, 1, 40, st[1])
    assert one.run() == 16  # alone
    torch.cuda.synchronize()
    alone = one.chi.cpu().numpy()
    volume = Call(256, 64, 2, 4000, st[0])  # over 0.1 s
    same = Call(256, 1, 1, 40, st[0])
    assert volume.run() == 4
    assert one.run() == 4
    assert same.run() == 16  # behind the volume on its stream: only `one` is beside it
    torch.cuda.synchronize()
    assert one.run() == 16  # alone again
    assert np.array_equal(alone, one.close()) and np.array_equal(alone, same.close())
    got = volume.close()
    f, m = volume.f[:1].contiguous(), volume.m[:1].contiguous()
    chi = torch.empty_like(f)
    ctx = pcs.pcs_create(256, 256, 1)
    pcs.pcs_solve_slices(ctx, f, m, 5e-4, STEP, STEP, 4000, chi)
    torch.cuda.synchronize()
    pcs.pcs_destroy(ctx)
    assert np.array_equal(got[:1], chi.cpu().numpy())


@pytest.mark.parametrize("H", [64, 128, 192, 256, 384, 512])
def test_contexts_in_flight_together(H):
    """Contexts of every shape at once, several slices each, two rounds: bit for bit the first one alone."""
    st = [torch.cuda.Stream() for _ in range(6)]
    S = 12 if H >= 384 else 24
    calls = [Call(H, S, 3, 30, s, use_graph=k == 2) for k, s in enumerate(st)]
    calls[0].run()
    torch.cuda.synchronize()
    ref = calls[0].chi.cpu().numpy()
    for _ in range(2):
        for c in calls:
            c.run()
    for c in calls:
        assert np.array_equal(ref, c.close())


def test_capture_by_the_caller_beside_other_solves():
    """A solve captured in the caller's graph while another context's solve runs: not disturbed, and replayed."""
    st = [torch.cuda.Stream() for _ in range(2)]
    one, volume = Call(256, 2, 1, 40, st[1]), Call(256, 64, 2, 2000, st[0])
    one.run()
    torch.cuda.synchronize()
    ref = one.chi.cpu().numpy()
    volume.run()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st[1]):
        assert one.run() == 16  # by the slice count: what is in flight now is not in flight at a replay
    torch.cuda.synchronize()
    one.chi.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(ref, one.chi.cpu().numpy())
    volume.close()
    one.close()


def test_solves_beside_another_threads_capture():
    """While this thread captures a graph of its own (global mode), another thread's solves look at what is
    in flight: they run, and the capture is not invalidated."""
    st = [torch.cuda.Stream() for _ in range(3)]
    volume, one = Call(256, 64, 2, 2000, st[0]), Call(256, 1, 1, 40, st[1])
    x = torch.zeros(64, device="cuda")
    volume.run()
    one.run()
    torch.cuda.synchronize()
    ref = volume.chi.cpu().numpy(), one.chi.cpu().numpy()
    g = torch.cuda.CUDAGraph()
    with ThreadPoolExecutor(1) as ex:
        with torch.cuda.graph(g, stream=st[2], capture_error_mode="global"):
            x.add_(1.0)
            assert ex.submit(lambda: (volume.run(), one.run())).result() == (4, 4)
            x.add_(1.0)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert x.cpu().tolist() == [2.0] * 64
    assert np.array_equal(ref[0], volume.close()) and np.array_equal(ref[1], one.close())
