"""Two host threads, each with contexts of its own object on its own stream,
build models at the same time: the shared memory that one object's kernels ask
for does not take away the other's.  Rows are those of a build alone."""
import threading

import numpy as np
import pytest

from paper_2002_12471_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def test_objects_of_different_size_in_two_threads():
    import torch

    import paper_2002_12471_gb300.lmosem as L
    dev = torch.device("cuda:0")
    jobs = []
    for n, angles, count in ((33, 4, 4 * 20), (96, 2, 2 * 20), (64, 3, 3 * 3000)):
        ph = S.brain_phantom(n, 256.0 / n)
        g = S.geometry(angles, n, 256.0 / n, 150.0, angle0_rad=0.1)
        ev = S.simulate_events(ph, g, count, seed=n, batch=1 << 16)
        jobs.append((ph, g, [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]))
    edges = np.linspace(100.0, 175.0, 4)

    def rows(job, stream, binned):
        ph, g, t = job
        with torch.cuda.stream(stream):
            ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=stream)
            try:
                if binned:
                    c = torch.zeros((g["n_angles"], g["n_bins"], 3), dtype=torch.float32, device=dev)
                    c[:, ::8] = 1.0
                    L.lmosem_build_model_binned(ctx, c, edges, 1)
                else:
                    L.lmosem_build_model(ctx, *t, 1)
                out = torch.zeros((20, L.lmosem_n_support(ctx)), dtype=torch.float32, device=dev)
                L.lmosem_model_rows(ctx, torch.arange(20, device=dev), out)
                stream.synchronize()
                return out
            finally:
                L.lmosem_destroy(ctx)

    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    want = [[rows(j, s, b) for b in (False, True)] for j, s in zip(jobs, streams)]
    failures = []

    def work(k):
        try:
            for i in range(150):
                if not torch.equal(rows(jobs[k], streams[k], i & 1), want[k][i & 1]):
                    failures.append("rows of thread %d" % k)
                    return
        except Exception as e:  # noqa: BLE001 - reported by the test
            failures.append(repr(e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
