"""Contexts of several host threads side by side, each with its own stream and a
mesh of its own size: a call takes nothing from the calls of another thread (the
dynamic shared memory that a kernel may take is an attribute of the function,
which all threads share).  The results are those of the same calls alone, bit
for bit."""
import threading

import pytest

from paper_2606_09275_gb300 import inputs
from test_gpu_resident_solve import MESHES, config

pytestmark = pytest.mark.gpu


def test_threads_of_different_meshes():
    import torch
    from paper_2606_09275_gb300 import mpm

    def job(key):
        cfg = config(*MESHES[key])
        ctx = mpm.Context()
        pts = inputs.make_points(cfg)
        P = mpm.Points(pts, capacity=12 * len(pts["x"]) + 400000)
        mesh = mpm.octree_build(ctx, cfg, P, body_z=inputs.body_z(cfg, 1) if cfg["body"] else None)
        n = 3 * mesh.info()["ndof"]
        zero = torch.zeros(n, dtype=torch.float64, device="cuda")
        g = torch.Generator(device="cuda").manual_seed(4)
        rhs = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        K = mpm.assemble(ctx, mesh, cfg, zero)["K"]

        def call(b=rhs):  # (P: the points live as long as the mesh)
            return mpm.solve(ctx, mesh, cfg, K, b, method=1, tol=1e-6)[0], P

        return call, zero

    keys = ["punch"] + ["few_quads"] * 4
    streams, jobs, want = [], [], []
    for k in keys:
        streams.append(torch.cuda.Stream())
        with torch.cuda.stream(streams[-1]):
            jobs.append(job(k))
            want.append(jobs[-1][0]()[0])
    torch.cuda.synchronize()
    errors, stop = [], threading.Event()

    def work(i):
        # (a solve for zero is over after one exchange: the launches follow closely)
        call, zero = jobs[i]
        try:
            with torch.cuda.stream(streams[i]):
                for k in range(4000 if i == 0 else 10 ** 9):
                    if stop.is_set():
                        break
                    if k % 50:
                        call(zero)
                    else:
                        assert torch.equal(call()[0], want[i])
        except BaseException as e:  # noqa: B902
            errors.append((keys[i], e))
        finally:
            if i == 0 or errors:
                stop.set()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(keys))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
