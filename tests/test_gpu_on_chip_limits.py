"""On-chip loops at the limits of their bookkeeping: checkpointed solves whose runs of stores and
reversals exceed what one launch lists, and several handles at once on streams of their own."""
import threading

import numpy as np
import pytest
import torch

from paper_2304_04781_gb300 import inputs

from .helpers import cuda, setup, solver
from .test_gpu_brick import both, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots,nt", [(31, 40), (33, 40), (70, 90), (70, 200)])
def test_more_checkpoints_than_a_launch_lists(slots, nt, monkeypatch):
    """A launch stores or reverses 32 states at most: 70 slots take three, on the way out and on
    the way back; the same bits as streaming."""
    shape = (8, 12, 20)
    prob, c, _ = setup(shape, nt, 1, seed=5)
    cc, rng = cuda(c), np.random.default_rng(3)
    d_obs = cuda(rng.standard_normal((nt + 1, prob.nrec, 3)) * 1e-6)
    dc = cuda(rng.standard_normal(shape))

    def run(s):
        J, g = s.gradient(cc, d_obs)
        return [J, g, s.hessvec(dc), s.stats()["forward_steps"]]

    same(*both(monkeypatch, lambda: solver(prob, storage="revolve", n_checkpoints=slots), run))


def test_handles_on_streams_of_their_own():
    """Four threads, a handle and a stream each: on-chip loops, prior solves and two-step passes
    at once give what they give alone."""
    jobs = [((32, 32, 32), {"storage": "full"}, 120), ((64, 64, 64), {"storage": "ae", "codec": "time"}, 48),
            ((96, 96, 96), {"storage": "revolve", "n_checkpoints": 5}, 40), ((160, 112, 112), {"storage": "full"}, 16)]
    Wt = inputs.codec_init(seed=4, n_hid=1024, n_lat=512)

    def work(job, n, out):
        try:
            shape, kw, nt = job
            with torch.cuda.stream(torch.cuda.Stream()):
                prob, c, _ = setup(shape, nt, 16, seed=5)
                s, cc = solver(prob, **kw), cuda(c)
                if kw["storage"] == "ae":
                    s.codec_set(Wt)
                d_obs = s.forward(cc) * 0.5
                for _ in range(n):
                    J, g = s.gradient(cc, d_obs)
                    x, it = s.prior_solve(cc, 1.0, 2.0 * prob.h ** 2)
                torch.cuda.current_stream().synchronize()
                out.append((J, g, x, it))
        except Exception as e:   # a thread's failure is the test's
            out.append(e)

    alone = []
    for job in jobs:
        out = []
        work(job, 1, out)
        alone.append(out[0])
    outs = [[] for _ in jobs]
    threads = [threading.Thread(target=work, args=(job, 6, out)) for job, out in zip(jobs, outs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, (b,) in zip(alone, outs):
        assert not isinstance(b, Exception), b
        assert a[0] == b[0] and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2]) and a[3] == b[3]
