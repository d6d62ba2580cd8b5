"""The fused update kernels against the same update on the FP32 CUDA cores (update_gemm 1, itself compared with
the FP64 oracle): the parameter change of one A2C step and of a PPO epoch, per network, at the edges of the 128-row
tile, of a chunk (whole rounds of tiles over the SMs) and of the input, hidden and output widths that each kernel
holds.  Tolerance: the oracle tests' 1e-4 of the largest gradient (two paths, each within it: 2e-4), and the half
ulp of a parameter that each SGD step can lose."""
import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W

pytestmark = pytest.mark.gpu
LR = 1.0


def _step(gemm, algo, env, h, n, T, dim, agents):
    kw = dict(dim=dim, n_gauss=64) if env == W.WS_ENV_LANDSCAPE else {}
    r = W.Rollout(env, W.WS_PATH_BATCHED_FP32, n, T, 9, h, h, param_seed=5,
                  flags=W.WS_FLAG_TRAIN | W.WS_FLAG_BOUNDS_CHECK, agents_per_env=agents, **kw)
    r.set_launch(update_gemm=gemm)
    r.reset(6)
    r.rollout(T)
    od, no = r.obs_dim(), r.n_out()
    nets = [(od, no)] + ([(16, 10)] if env == W.WS_ENV_ECONOMY else [])
    count = lambda a, b: a * h + h + h * h + h + h * b + b  # noqa: E731
    sizes = {W.WS_F_PARAMS: [count(*s) for s in nets], W.WS_F_CRITIC: [count(s[0], 1) for s in nets]}
    get = lambda: [r.fetch_raw(f, 4 * sum(s)).view(np.float32).copy() for f, s in sizes.items()]  # noqa: E731
    before = get()
    if algo == "a2c":
        r.a2c_update(T, LR, 0.5, 0.01)
    else:
        r.advantages(T)
        r.ppo_update(T, LR, 0.2, 0.5, 0.01)
    r.sync()
    after = get()
    adv = r.fetch(W.WS_F_ADVANTAGE, 0, T) if algo == "ppo" else None
    r.close()
    cuts = [np.cumsum(s)[:-1] for s in sizes.values()]
    return [np.split(b, c) for b, c in zip(before, cuts)], [np.split(a, c) for a, c in zip(after, cuts)], adv


CASES = [
    ("a2c", W.WS_ENV_CONTROL, 64, 1, 1, 0), ("a2c", W.WS_ENV_CONTROL, 256, 127, 1, 0),
    ("ppo", W.WS_ENV_CONTROL, 128, 129, 1, 0), ("a2c", W.WS_ENV_CONTROL, 128, 5000, 14, 0),
    ("ppo", W.WS_ENV_ACROBOT, 256, 300, 7, 0), ("a2c", W.WS_ENV_ACROBOT, 128, 641, 3, 0),
    ("ppo", W.WS_ENV_ECONOMY, 64, 5, 3, 0), ("a2c", W.WS_ENV_ECONOMY, 256, 9, 2, 0),
    ("ppo", W.WS_ENV_ECONOMY, 128, 40, 14, 0),
    ("a2c", W.WS_ENV_LANDSCAPE, 64, 200, 2, 5), ("ppo", W.WS_ENV_LANDSCAPE, 128, 333, 3, 10),
    ("ppo", W.WS_ENV_LANDSCAPE, 256, 700, 2, 24), ("a2c", W.WS_ENV_LANDSCAPE, 256, 130, 2, 1),
]


@pytest.mark.parametrize("algo,env,h,n,T,dim", CASES)
def test_fused_update_equals_cuda_core_update(algo, env, h, n, T, dim):
    agents = np.random.default_rng(2).integers(2, 200, n) if env == W.WS_ENV_ECONOMY else None
    b0, a0, adv0 = _step(0, algo, env, h, n, T, dim, agents)
    b1, a1, adv1 = _step(1, algo, env, h, n, T, dim, agents)
    for field in range(2):
        for pb0, pa0, pb1, pa1 in zip(b0[field], a0[field], b1[field], a1[field]):
            assert np.array_equal(pb0, pb1)
            g0, g1 = pb0.astype(np.float64) - pa0, pb1.astype(np.float64) - pa1
            tol = 2e-4 * np.abs(g1).max() + 1.2 * np.spacing(np.maximum(np.abs(pa1), np.abs(pb1)))
            assert np.abs(g1).max() > 0
            assert np.all(np.abs(g0 - g1) <= tol), np.abs(g0 - g1).max()
    if adv0 is not None:  # the critic's values, within the products' error at the values' scale
        assert np.abs(adv0 - adv1).max() <= 1e-4 * max(1.0, np.abs(adv1).max())
