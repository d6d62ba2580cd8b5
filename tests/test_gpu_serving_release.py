"""Releasing a request with chunks in flight: the wait for its kernels holds no other client up, its bytes are free
when the call returns, and a server that closes meanwhile waits for it."""
import threading
import time

import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu
GB = 1 << 30


def busy_request(srv):
    """A request with one 200-step chunk (some 75 ms) running and a second one behind it."""
    q, keep = W.make_request(W.WS_ENV_CONTROL, W.WS_PATH_BATCHED_FP32, 131072, 2000, 200, 500, 256, 256, seed=3)
    st, rid = srv.submit(q)
    assert st == W.WS_OK
    assert srv.wait_chunk(rid, 0, 60000) == W.WS_OK
    assert srv.ack(rid, 0) == W.WS_OK
    return rid


def test_release_does_not_hold_the_server():
    need_gpu()
    srv = W.Server(6 * GB)
    rid = busy_request(srv)
    took = []

    def release():
        t = time.perf_counter()
        assert srv.release(rid) == W.WS_OK
        took.append(time.perf_counter() - t)
    th = threading.Thread(target=release)
    th.start()
    longest, waits = 0.0, 0
    while not took:
        t = time.perf_counter()
        srv.stats()
        longest = max(longest, time.perf_counter() - t)
        waits += 1
        time.sleep(1e-3)
    th.join()
    assert srv.stats()["used_bytes"] == 0
    # the release had kernels to wait for; the other client's calls went on meanwhile
    assert took[0] > 0.02 and longest < took[0] / 4, (took[0], longest, waits)
    assert srv.wait_chunk(rid, 1, 1000) == W.WS_ERR_INVALID
    assert srv.release(rid) == W.WS_ERR_INVALID
    srv.close()


def test_close_waits_for_a_release():
    need_gpu()
    srv = W.Server(6 * GB)
    rid = busy_request(srv)
    got = []
    th = threading.Thread(target=lambda: got.append(srv.release(rid)))
    th.start()
    while srv.stats()["active"] and not got:  # the release has begun (or ended)
        time.sleep(1e-3)
    srv.close()
    th.join()
    assert got == [W.WS_OK]
