"""The fused FP32 classic-control kernel against the plain path's per-sub-step kernels: every record, the final
state and the last logits byte for byte (the arithmetic is the same, operation by operation; the plain path is
itself compared with the FP64 oracle).  Widths on both sides of each tile (64, 128, 256 units, odd ones, zero
padding of K and N), env counts at the edges of each row tile, launches that cross a chunk and the ring's end."""
import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W

pytestmark = pytest.mark.gpu


def _records(env, path, n, T, h0, h1, ring):
    r = W.Rollout(env, path, n, ring, 13, h0, h1, param_seed=3, chunk_steps=7 if path else 0,
                  flags=W.WS_FLAG_DEBUG_LOGITS | W.WS_FLAG_BOUNDS_CHECK)
    r.reset(11)
    r.rollout(T - 1)
    r.step()
    r.sync()
    fields = (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP, W.WS_F_REWARD, W.WS_F_DONE, W.WS_F_POLICY_OUT)
    out = [r.fetch(f, T - ring, ring) for f in fields]
    out += [r.fetch_raw(W.WS_F_STATE, 20 * n), r.fetch_raw(W.WS_F_LOGITS, 4 * n * r.n_out())]
    r.close()
    return out


@pytest.mark.parametrize("env", [W.WS_ENV_CONTROL, W.WS_ENV_ACROBOT])
@pytest.mark.parametrize("h0,h1", [(64, 64), (5, 3), (128, 128), (100, 37), (256, 256), (37, 250), (130, 64)])
def test_fused_fp32_equals_plain(env, h0, h1):
    # one env; partial tiles; the env counts around which the row tile changes (8, 16 and 32 envs per SM)
    for n in (1, 77, 1216, 1217, 2433, 4865, 31000):
        T, ring = (40, 30) if n < 5000 else (3, 2)
        a = _records(env, W.WS_PATH_PLAIN_FP32, n, T, h0, h1, ring)
        b = _records(env, W.WS_PATH_BATCHED_FP32, n, T, h0, h1, ring)
        for i, (x, y) in enumerate(zip(a, b)):
            assert np.array_equal(x.view(np.uint8), y.view(np.uint8)), (n, i)


@pytest.mark.parametrize("h0,h1", [(61, 33), (37, 100), (130, 253)])
def test_infinite_state_stays_in_its_row(h0, h1):
    # an infinite observation against a unit past the width (a zero weight) must not reach the units there are
    for n in (77, 31000):
        rows = []
        for path in (W.WS_PATH_PLAIN_FP32, W.WS_PATH_BATCHED_FP32):
            r = W.Rollout(W.WS_ENV_CONTROL, path, n, 4, 13, h0, h1, param_seed=3, flags=W.WS_FLAG_DEBUG_LOGITS)
            r.reset(11)
            state = r.fetch_raw(W.WS_F_STATE, 20 * n).copy()
            state[:16 * n].view(np.float32).reshape(4, n)[0, 5] = np.inf
            r.load_raw(W.WS_F_STATE, state, k=0)
            r.rollout(4)
            r.sync()
            rows.append([r.fetch(f, 0, 4) for f in (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP, W.WS_F_POLICY_OUT)])
            r.close()
        assert np.isinf(rows[0][0]).any() and np.isfinite(rows[0][3]).all()
        for x, y in zip(*rows):
            assert np.array_equal(x.view(np.uint8), y.view(np.uint8)), n
