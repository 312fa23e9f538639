"""The server's steps by the kinds of requests they hold (thread kernel, warp
kernel pair by pair, line by line): kinds that come, go and come back between
steps, alone and together, with few items and with more than a thousand.  Every
image is bitwise the one a server of that request alone gives."""
import numpy as np
import pytest

from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_serve_gpu import run_alone, submit

pytestmark = pytest.mark.gpu

# (sources, domains, ROI side): thread, pairs, lines
KINDS = {"t": (5, 3, 50), "p": (20, 12, 40), "l": (60, 30, 30),
         "T": (2, 2, 400), "P": (3, 8, 400)}


def _requests(word):
    out = []
    for i, c in enumerate(word):
        S, M, n = KINDS[c]
        r = W.serving_requests(1, seed=50 + i, max_src=1, max_mosaic=1)[0]
        r.umats = W.mosaic_umats(np.random.default_rng(i), M, 0.05)
        _, r.lambdas, r.weights = W.gaussian_spectrum(S, 9.5, 0.005)
        r.roi = (900 + 10 * i, 1100, n, n)
        out.append(r)
    return out


@pytest.mark.parametrize("word", ["tlptlp", "lllttpl", "TtPpl", "pPlTt"])
def test_kinds_come_and_go(word):
    base = W.serving_detector_shot()
    reqs = _requests(word)
    alone = run_alone(base, reqs)
    srv = nbgb.Server(base, max_slots=4, pool_bytes=16 << 20)
    # one after another, then all of them at once
    for r, a in zip(reqs, alone):
        rid = submit(srv, r)
        srv.run_all()
        assert np.array_equal(srv.result(rid), a)
    ids = [submit(srv, r) for r in reqs]
    done = srv.run_all()
    assert sorted(done) == sorted(ids)
    for rid, a in zip(ids, alone):
        assert np.array_equal(srv.result(rid), a)
    srv.close()
    # and by steps of a few items, with requests that arrive in between
    srv = nbgb.Server(base, max_slots=3, pool_bytes=16 << 20,
                      step_budget=300000)
    ids = []
    for r in reqs:
        ids.append(submit(srv, r))
        srv.step()
    srv.run_all()
    for rid, a in zip(ids, alone):
        assert np.array_equal(srv.result(rid), a)
    srv.close()
