"""Host threads with handles of different sizes: a kernel's shared-memory limit
belongs to the function on the device, so one thread's call must not lower it
under the launch of another."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


def run_threads(work):
    """Runs work[i]() in a thread each, started together; returns what they raised."""
    start, raised = threading.Barrier(len(work)), []

    def body(f):
        try:
            start.wait()
            f()
        except Exception as e:  # noqa: BLE001
            raised.append(repr(e))

    threads = [threading.Thread(target=body, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return raised


def images(W, H, seed):
    rng = np.random.default_rng(seed)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    return torch.from_numpy(left).cuda(), torch.from_numpy(np.roll(left, -5, axis=1).copy()).cuda()


@pytest.mark.parametrize("cost, window", [(sgm.SGM_COST_CENSUS, 5), (sgm.SGM_COST_SAD, 7)])
def test_handles_of_two_widths_on_two_threads(cost, window):
    # The narrow rows need less shared memory in the winner-takes-all kernel, the
    # smaller D in the SAD kernel, and both run the same instance of it.
    p = sgm.SgmParams(census_w=window, census_h=window, path_mask=sgm.SGM_PATHS_4, P1=8, P2=32, lr_tolerance=1,
                      median_k=3, cost=cost)
    work, outs = [], []
    for W, D in ((8000, 128), (160, 90)):
        h = sgm.Handle(W, 2, D, p)
        L, R = images(W, 2, W)
        want, disp = (torch.empty((2, W), dtype=torch.uint8, device="cuda") for _ in range(2))
        h.compute(L, R, want)
        torch.cuda.synchronize()
        outs.append((want, disp, h))
        stream = torch.cuda.Stream()

        def many(h=h, L=L, R=R, disp=disp, stream=stream):
            for _ in range(4000):
                h.compute(L, R, disp, stream)
            stream.synchronize()

        work.append(many)
    assert run_threads(work) == []
    for want, disp, _ in outs:
        assert torch.equal(want, disp)


def test_batches_of_two_sizes_on_many_threads():
    # one shared aggregation launch each, whose shared memory grows with the pairs;
    # changing outputs make every run capture it anew
    p = sgm.SgmParams(census_w=5, census_h=5, path_mask=sgm.SGM_PATHS_4, P1=8, P2=32, lr_tolerance=1, median_k=3)
    work, outs = [], []
    for n in (24, 2, 2, 2, 2, 2, 2):
        b = sgm.Batch([(48, 16, 32)] * n, p)
        b.set_tuning(1, 2)
        ins = [images(48, 16, i) for i in range(n)]
        Ls, Rs = [i[0] for i in ins], [i[1] for i in ins]
        disps = [[torch.empty((16, 48), dtype=torch.uint8, device="cuda") for _ in range(n)] for _ in range(3)]
        b.run(Ls, Rs, disps[2])
        torch.cuda.synchronize()
        outs.append((b, disps))
        stream = torch.cuda.Stream()

        def many(b=b, Ls=Ls, Rs=Rs, disps=disps, stream=stream):
            for i in range(400):
                b.run(Ls, Rs, disps[i % 2], stream=stream)
                stream.synchronize()

        work.append(many)
    assert run_threads(work) == []
    for b, disps in outs:
        for k in range(2):
            assert all(torch.equal(a, c) for a, c in zip(disps[k], disps[2]))
        b.close()
