"""Two chunks of a request in flight and a client that reads and acknowledges late: the records are a plain roll-out's,
and no chunk is overwritten before it is acknowledged."""
import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu
FIELDS = (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP, W.WS_F_REWARD, W.WS_F_DONE)


@pytest.mark.parametrize("path", [W.WS_PATH_BATCHED_FP32, W.WS_PATH_BATCHED_BF16])
def test_late_acknowledgements(path):
    need_gpu()
    n, horizon, chunk = 700, 330, 50  # seven chunks, the last of 30 steps
    r = W.Rollout(W.WS_ENV_CONTROL, path, n, horizon, 60, 64, 64, param_seed=5, chunk_steps=chunk)
    r.rollout(horizon)
    ref = [r.fetch(f, 0, horizon) for f in FIELDS]
    r.close()
    srv = W.Server(256 << 20)
    q, keep = W.make_request(W.WS_ENV_CONTROL, path, n, horizon, chunk, 60, 64, 64, seed=5)
    st, rid = srv.submit(q)
    assert st == W.WS_OK

    def read(c):
        for f, a in zip(FIELDS, ref):
            want = np.ascontiguousarray(a[c * chunk:(c + 1) * chunk])
            got = np.empty_like(want)
            assert srv.fetch(rid, f, c, got) == W.WS_OK
            assert np.array_equal(got.view(np.uint8), want.view(np.uint8)), (c, f)
    for c in (0, 2, 4):  # the second of two chunks read first; both acknowledged at once
        assert srv.wait_chunk(rid, c + 1, 30000) == W.WS_OK
        assert srv.wait_chunk(rid, c + 2, 50) == W.WS_ERR_TIMEOUT  # its ring half is not free
        read(c + 1)
        read(c)
        assert srv.ack(rid, c + 1) == W.WS_OK
        assert srv.fetch(rid, W.WS_F_DONE, c, np.empty(n * chunk, np.uint8)) == W.WS_ERR_RANGE
    assert srv.wait_chunk(rid, 6, 30000) == W.WS_OK
    read(6)
    assert srv.ack(rid, 6) == W.WS_OK and srv.release(rid) == W.WS_OK
    srv.close()
