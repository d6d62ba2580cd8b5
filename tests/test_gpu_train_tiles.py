"""The fused update's row tiles against the FP32 CUDA-core update (update_gemm 1), tolerances as in
test_gpu_train_tc.py."""
import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu
from tests.refuse_launch import child

pytestmark = pytest.mark.gpu
LR = 1.0


def _nets(r, env, h):
    nets = [(r.obs_dim(), r.n_out())] + ([(16, 10)] if env == W.WS_ENV_ECONOMY else [])
    count = lambda a, b: a * h + h + h * h + h + h * b + b  # noqa: E731
    return {W.WS_F_PARAMS: [count(*s) for s in nets], W.WS_F_CRITIC: [count(s[0], 1) for s in nets]}


def _step(gemm, algo, env, h, n, T, dim, agents=None, change=None):
    kw = dict(dim=dim, n_gauss=64) if env == W.WS_ENV_LANDSCAPE else {}
    r = W.Rollout(env, W.WS_PATH_BATCHED_FP32, n, T, 9, h, h, param_seed=5,
                  flags=W.WS_FLAG_TRAIN | W.WS_FLAG_BOUNDS_CHECK, agents_per_env=agents, **kw)
    r.set_launch(update_gemm=gemm)
    sizes = _nets(r, env, h)
    get = lambda: [r.fetch_raw(f, 4 * sum(s)).view(np.float32).copy() for f, s in sizes.items()]  # noqa: E731
    if change:
        for f, p in zip(sizes, get()):
            change(p)
            r.load_raw(f, p.view(np.uint8))
    r.reset(6)
    r.rollout(T)
    before = get()
    if algo == "a2c":
        r.a2c_update(T, LR, 0.5, 0.01)
    else:
        r.advantages(T)
        r.ppo_update(T, LR, 0.2, 0.5, 0.01)
    r.sync()
    after = get()
    r.close()
    cuts = [np.cumsum(s)[:-1] for s in sizes.values()]
    return [np.split(b, c) for b, c in zip(before, cuts)], [np.split(a, c) for a, c in zip(after, cuts)]


def _compare(algo, env, h, n, T, dim, agents=None, change=None):
    b0, a0 = _step(0, algo, env, h, n, T, dim, agents, change)
    b1, a1 = _step(1, algo, env, h, n, T, dim, agents, change)
    for field in range(2):
        for pb0, pa0, pb1, pa1 in zip(b0[field], a0[field], b1[field], a1[field]):
            assert np.array_equal(pb0, pb1)
            ok = np.isfinite(pa1)
            assert np.array_equal(pa0[~ok], pa1[~ok]) and ok.sum() >= ok.size - 1  # the one that was set
            pb, p0, p1 = pb0[ok].astype(np.float64), pa0[ok], pa1[ok]
            g0, g1 = pb - p0, pb - p1
            tol = 2e-4 * np.abs(g1).max() + 1.2 * np.spacing(np.maximum(np.abs(p1), np.abs(pb0[ok])))
            assert np.abs(g1).max() > 0
            assert np.all(np.abs(g0 - g1) <= tol), np.nanmax(np.abs(g0 - g1))


@pytest.mark.parametrize("algo,env,h,n,T,dim", [
    ("a2c", W.WS_ENV_CONTROL, 64, 129, 1, 0), ("ppo", W.WS_ENV_CONTROL, 256, 1, 1, 0),
    ("a2c", W.WS_ENV_ACROBOT, 128, 200, 2, 0), ("a2c", W.WS_ENV_LANDSCAPE, 64, 130, 2, 9)])
def test_infinite_weight_and_a_partial_tile(algo, env, h, n, T, dim):
    # an infinite first-layer weight saturates its unit in every recorded row (no observation is zero); the rows
    # past the end of the last tile must not turn it into a NaN
    def change(p):
        p[5] = np.inf
    _compare(algo, env, h, n, T, dim, change=change)


def advantage_launches(rt):
    r = W.Rollout(W.WS_ENV_CONTROL, W.WS_PATH_BATCHED_FP32, 100, 4, 9, 256, 256, flags=W.WS_FLAG_TRAIN)
    r.reset(1)
    r.rollout(4)
    rt.refuse_launch(-1)
    r.advantages(4)
    assert rt.launches_seen() == 4  # returns, the forward's weight image, the forward, the store
    r.close()


def test_advantages_pack_for_the_forward_alone(tmp_path):
    need_gpu()
    child("advantage_launches", tmp_path, module="test_gpu_train_tiles")


@pytest.mark.parametrize("algo,env,h,n,T,dim", [
    ("ppo", W.WS_ENV_LANDSCAPE, 256, 8191, 9, 24), ("a2c", W.WS_ENV_LANDSCAPE, 256, 8191, 9, 16),
    ("ppo", W.WS_ENV_LANDSCAPE, 64, 8191, 9, 10), ("a2c", W.WS_ENV_ECONOMY, 256, 150, 4, 0)])
def test_many_tiles_without_an_output_layer(algo, env, h, n, T, dim):
    # several tiles of each network per CTA, two chunks with a partial last tile, where the output layer, or its
    # gradients, are formed outside the fused kernels (and at 256 units dW1 is summed in global memory)
    agents = np.random.default_rng(2).integers(100, 200, n) if env == W.WS_ENV_ECONOMY else None
    _compare(algo, env, h, n, T, dim, agents)
