"""Roll-outs of a single chunk, which are launched directly or through a graph: the same answers either way."""
import ctypes

import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu
from tests.refuse_launch import child

pytestmark = pytest.mark.gpu

# env, path, hidden width, extra configuration: the paths whose chunk is one launch
SHAPES = [(W.WS_ENV_CONTROL, W.WS_PATH_BATCHED_BF16, 64, {}), (W.WS_ENV_ACROBOT, W.WS_PATH_BATCHED_BF16, 64, {}),
          (W.WS_ENV_CONTROL, W.WS_PATH_BATCHED_FP32, 64, {}), (W.WS_ENV_ACROBOT, W.WS_PATH_BATCHED_FP32, 64, {}),
          (W.WS_ENV_ECONOMY, W.WS_PATH_BATCHED_BF16, 128, {}),
          (W.WS_ENV_LANDSCAPE, W.WS_PATH_BATCHED_BF16, 256, dict(dim=8, n_gauss=256))]


@pytest.mark.parametrize("env,path,h,kw", SHAPES)
def test_a_capturing_stream_takes_no_rollout(env, path, h, kw):
    # its steps would be counted without having run; refused whether or not its graph is there already
    torch = need_gpu()
    rt = ctypes.CDLL("libcudart.so.13")
    for warm in (0, 1, 20):
        for mode in (0, 1, 2):
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                r = W.Rollout(env, path, 30, 40, 15, h, h, **kw)
                r.reset(3)
                for _ in range(warm):
                    r.rollout(10)
                torch.cuda.synchronize()
                k, g = r.k, ctypes.c_void_p()
                assert rt.cudaStreamBeginCapture(ctypes.c_void_p(st.cuda_stream), mode) == 0
                got = W.ws_rollout(r.ctx, 10)
                rt.cudaStreamEndCapture(ctypes.c_void_p(st.cuda_stream), ctypes.byref(g))
                rt.cudaGetLastError()
                if g.value:
                    rt.cudaGraphDestroy(g)
                assert got == W.WS_ERR_CUDA and r.k == k, (warm, mode)
                r.close()
    torch.cuda.synchronize()


def count_launches(rt):
    """Kernels launched one by one (not by a graph) in each of equal roll-outs, whose records are the same."""
    fields = (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP, W.WS_F_REWARD, W.WS_F_DONE)
    for env, path, h, kw in SHAPES:
        r = W.Rollout(env, path, 300, 40, 15, h, h, **kw)
        seen, records = [], set()
        for _ in range(4):
            r.reset(3)
            rt.refuse_launch(-1)
            r.rollout(10)
            seen.append(rt.launches_seen())
            records.add(b"".join(r.fetch(f, 0, 10).tobytes() for f in fields))
        # launched directly once (no capture), captured (the launches are seen again), then through the graph
        assert seen == [2, 2, 0, 0] and len(records) == 1, (env, path, seen)
        r.reset(4)  # another seed: begins anew
        rt.refuse_launch(-1)
        r.rollout(10)
        assert rt.launches_seen() == 2
        r.close()


def test_repeated_rollouts_go_through_a_graph(tmp_path):
    need_gpu()
    child("count_launches", tmp_path, module="test_gpu_short_rollouts")


def many_lengths(rt):
    r = W.Rollout(W.WS_ENV_CONTROL, W.WS_PATH_BATCHED_FP32, 9, 40, 15, 64, 64, chunk_steps=5)
    r.reset(3)
    for n in range(6, 106):
        r.rollout(n)
    r.sync()
    rt.refuse_launch(-1)
    r.rollout(105)
    assert rt.launches_seen() == 0  # a late one: still there
    r.rollout(6)
    assert rt.launches_seen() == 3  # an early one: captured again (two chunks and the step count)
    r.sync()
    ref = W.Rollout(W.WS_ENV_CONTROL, W.WS_PATH_PLAIN_FP32, 9, 40, 15, 64, 64)
    ref.reset(3)
    ref.rollout(r.k)
    for f in (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP):
        assert r.fetch(f, r.k - 40, 40).tobytes() == ref.fetch(f, r.k - 40, 40).tobytes()


def test_graphs_of_many_lengths_are_bounded(tmp_path):
    need_gpu()
    child("many_lengths", tmp_path, module="test_gpu_short_rollouts")


def served_graphs(rt):
    srv = W.Server(256 << 20)
    for path in (W.WS_PATH_BATCHED_FP32, W.WS_PATH_BATCHED_BF16):
        for horizon, chunks, graphs in ((50, 1, 0), (130, 3, 0), (150, 3, 1), (230, 5, 1)):
            before = rt.graphs_made()
            q, _keep = W.make_request(W.WS_ENV_CONTROL, path, 300, horizon, 50, 60, 64, 64, seed=5)
            st, rid = srv.submit(q)
            assert st == W.WS_OK
            for c in range(chunks):
                assert srv.wait_chunk(rid, c, 30000) == W.WS_OK and srv.ack(rid, c) == W.WS_OK
            assert rt.graphs_made() - before == graphs, (path, horizon)
            assert srv.release(rid) == W.WS_OK
    srv.close()


def test_served_requests_capture_what_comes_again(tmp_path):
    # three chunks of a length are the least for which a capture pays
    need_gpu()
    child("served_graphs", tmp_path, module="test_gpu_short_rollouts")
