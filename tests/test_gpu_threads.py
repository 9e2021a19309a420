"""Handles of their own in threads of their own: calls on two hierarchies of different basis
size at the same time, from two host threads on two streams, give the bits that each gives
alone.  Pairs whose launches share a kernel and need different amounts of shared memory: the
basis change and the panels (d = 100 and 125), whole items (60 and 64), all steps in one
launch (36 and 45), the gradient's contractions (100 and 125)."""
import threading

import numpy as np
import pytest

import workloads as W
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


def together(works):
    """Each work's results in its own thread, all started at once; raises what one raised."""
    out, errors, start = [None] * len(works), [], threading.Barrier(len(works))

    def body(i):
        try:
            start.wait(60)
            out[i] = works[i]()
        except Exception as e:   # noqa: BLE001 -- reported below
            errors.append(e)

    threads = [threading.Thread(target=body, args=(i,)) for i in range(len(works))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]
    return out


@pytest.mark.parametrize("levels,depth,branches,calls", [
    (((4, 5, 5), (5, 5, 5)), 0, 1, 1500),
    (((3, 5, 4), (4, 4, 4)), 1, 100, 150),
    (((3, 3, 4), (3, 3, 5)), 1, 1, 1500),
])
def test_two_hierarchies_at_once(levels, depth, branches, calls):
    torch = pytest.importorskip("torch")
    works, refs = [], []
    for lv in levels:
        h = H.heom_build_hierarchy(model_of(lv, depth))
        g = torch.Generator(device="cuda")
        g.manual_seed(sum(lv))
        x = torch.randn((branches, h.n_ado, h.d, h.d), generator=g, device="cuda", dtype=torch.complex128)
        y, a, b = (torch.empty_like(x) for _ in range(3))
        stream = torch.cuda.Stream()

        def work(h=h, x=x, y=y, a=a, b=b, stream=stream, n=calls):
            first = None
            with torch.cuda.stream(stream):
                bad = torch.zeros((), dtype=torch.int64, device="cuda")
                for _ in range(n):
                    y.copy_(x)
                    H.heom_propagate_dev(h, y.data_ptr(), a.data_ptr(), b.data_ptr(), branches, H.FP64, 0.25, 1,
                                         stream.cuda_stream)
                    if first is None:
                        first = y.clone()
                    bad += (y != first).any()
            stream.synchronize()
            return first.cpu().numpy(), int(bad)

        torch.cuda.synchronize()
        refs.append(work(n=1)[0])
        works.append(work)
    for ref, (first, bad) in zip(refs, together(works)):
        assert bad == 0 and np.array_equal(first, ref)


def test_two_gradients_at_once():
    grid = W.grid(0.25, 2, 2, 2, (0.0,), t_eq_fs=1.0)
    works, refs = [], []
    for lv in ((4, 5, 5), (5, 5, 5)):
        h = H.heom_build_hierarchy(model_of(lv, 0))
        eq = H.heom_equilibrate(h, 0.25, 1.0, 0.0)

        def work(h=h, eq=eq, n=4):
            return [H.heom_response_2d_grad(h, eq, grid, np.zeros((1, 2, 2)), 4) for _ in range(n)]

        refs.append(work(n=1)[0])
        works.append(work)
    for (loss, dtheta), got in zip(refs, together(works)):
        scale = np.abs(dtheta).max()
        for l, t in got:   # the gradient's sums end in atomic additions
            assert abs(l - loss) <= 1e-12 * abs(loss) and np.abs(t - dtheta).max() <= 1e-10 * scale
