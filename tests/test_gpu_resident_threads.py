"""Resident solves of several threads: those that fit on the chip together run side by
side, the others one after another, and all give what they give alone."""
import threading
import time

import numpy as np
import pytest
import torch

from paper_2408_03452_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_03452_gb300 import build, tpfa
    build.build()
    return tpfa


class _Job:
    def __init__(self, tp, shape, sigma, seed, **opts):
        nx, ny, nz = shape
        K = torch.from_numpy(synth.lognormal_field(nx, ny, nz, sigma, seed)).cuda()
        mask, pD = (torch.from_numpy(v).cuda() for v in synth.dirichlet_faces(nx, ny, nz, "x", 1.0, 0.0))
        self.ctx = tp.Context(*shape)
        for k, v in opts.items():
            self.ctx.set_option(k, v)
        self.coef, self.coef64 = self.ctx.build_trans(K, mask, None, 0.0)
        self.b = self.ctx.build_rhs(K, mask, None, pD)
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()

    def run(self, tol=1e-9, maxit=300000):
        with torch.cuda.stream(self.stream):
            x = torch.zeros_like(self.b)
            self.x, self.info = self.ctx.cg_solve(self.coef, self.coef64, self.b, x=x, tol=tol,
                                                  maxit=maxit, check=False)
        self.end = time.perf_counter()
        return self.x.cpu().numpy(), self.info["iters"]


def test_small_solve_does_not_wait_for_a_long_one(tp):
    """128 of the SMs hold a solve of a tenth of a second and more; one of 8 blocks runs
    beside it."""
    long = _Job(tp, (64, 64, 64), 4.0, 71, max_outer=1, inner_rtol=1e-12)
    short = _Job(tp, (32, 16, 8), 1.0, 72)
    want = short.run()
    t = threading.Thread(target=long.run)
    t.start()
    time.sleep(0.03)
    got = short.run()
    t.join()
    assert long.info["inner_ms"] > 100, long.info
    assert short.end < long.end
    assert got[1] == want[1] and np.array_equal(got[0], want[0])


def test_many_threads_agree_with_solves_alone(tp):
    """Six solves at once on their own streams: together they want more SMs than there
    are, so that some wait."""
    shapes = [(64, 64, 64), (33, 17, 9), (96, 96, 48), (40, 20, 12), (128, 128, 80), (32, 32, 32)]
    jobs = [_Job(tp, s, 1.0, 80 + i, precond=i % 2) for i, s in enumerate(shapes)]
    alone = [j.run() for j in jobs]
    got = [[] for _ in jobs]

    def repeat(i):
        for _ in range(5):
            got[i].append(jobs[i].run())

    threads = [threading.Thread(target=repeat, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, job in enumerate(jobs):
        assert job.info["code"] == 0
        for x, iters in got[i]:
            assert iters == alone[i][1] and np.array_equal(x, alone[i][0]), i
