"""Launches that the runtime refuses: each launch of a call in turn, in a process of its own with tests/refuse_launch.cpp
ahead of the library.  A call that lost a launch reports it, unless something took the launch's place: then what it
gives is right.

Updates: the parameter change is the undisturbed update's within the two paths' error (2e-4 of the largest gradient
and the half ulp of a parameter, as the fused update against the FP32 one), with the output layers in the fused
kernels and outside, over one chunk and two with a partial last tile."""
import ctypes

import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu
from tests.refuse_launch import child

pytestmark = pytest.mark.gpu
LR = 1.0

# algorithm, env, hidden width, envs, steps, dimension
UPDATES = [("a2c", W.WS_ENV_CONTROL, 128, 5000, 14, 0), ("ppo", W.WS_ENV_CONTROL, 64, 129, 2, 0),
           ("ppo", W.WS_ENV_LANDSCAPE, 128, 5000, 14, 9), ("a2c", W.WS_ENV_LANDSCAPE, 64, 130, 2, 5),
           ("ppo", W.WS_ENV_ECONOMY, 256, 5, 3, 0)]


def context(env, h, n, T, dim, flags=0, path=W.WS_PATH_BATCHED_FP32):
    kw = {}
    if env == W.WS_ENV_LANDSCAPE:
        kw.update(dim=dim, n_gauss=64)
    if env == W.WS_ENV_ECONOMY:
        kw["agents_per_env"] = np.random.default_rng(2).integers(100, 200, n)
    r = W.Rollout(env, path, n, T, 9, h, h, param_seed=5, flags=flags, **kw)
    r.reset(6)
    return r


def update(algo, env, h, n, T, dim, arm=lambda: None, disarm=lambda: None):
    """(status, before, after, advantages) of one update; arm() before its calls, disarm() after."""
    r = context(env, h, n, T, dim, W.WS_FLAG_TRAIN | W.WS_FLAG_BOUNDS_CHECK)
    r.rollout(T)
    nets = [(r.obs_dim(), r.n_out())] + ([(16, 10)] if env == W.WS_ENV_ECONOMY else [])
    count = lambda a, b: a * h + h + h * h + h + h * b + b  # noqa: E731
    sizes = {W.WS_F_PARAMS: sum(count(*s) for s in nets), W.WS_F_CRITIC: sum(count(s[0], 1) for s in nets)}
    get = lambda: [r.fetch_raw(f, 4 * s).view(np.float32).copy() for f, s in sizes.items()]  # noqa: E731
    before, adv = get(), None
    arm()
    if algo == "a2c":
        st = W.ws_a2c_update(r.ctx, T, LR, 0.5, 0.01)
    else:
        st = W.ws_advantages(r.ctx, T)
        if st == W.WS_OK:
            st = W.ws_ppo_update(r.ctx, T, LR, 0.2, 0.5, 0.01)
    disarm()
    if st != W.WS_OK:
        assert W.ws_last_error(r.ctx)
        r.close()
        return st, before, None, None
    r.sync()
    after = get()
    if algo == "ppo":
        adv = r.fetch(W.WS_F_ADVANTAGE, 0, T)
    r.close()
    return st, before, after, adv


def check(ref, got):
    for b, a, b2, a2 in zip(ref[1], ref[2], got[1], got[2]):
        assert np.array_equal(b, b2)
        g, g2 = b.astype(np.float64) - a, b.astype(np.float64) - a2
        tol = 2e-4 * np.abs(g).max() + 1.2 * np.spacing(np.maximum(np.abs(a), np.abs(b)))
        assert np.abs(g).max() > 0
        assert np.all(np.abs(g - g2) <= tol), (np.abs(g - g2).max(), np.abs(g).max())
    if ref[3] is not None:
        assert np.abs(ref[3] - got[3]).max() <= 1e-4 * max(1.0, np.abs(ref[3]).max())


# ---- in the process with the launch entries replaced: `rt` is that library
def refuse_updates(rt, case):
    ref = update(*case, arm=lambda: rt.refuse_launch(-1))
    assert ref[0] == W.WS_OK
    n, lost = rt.launches_seen(), 0
    assert n >= 8
    for i in range(n):
        got = update(*case, arm=lambda: rt.refuse_launch(i), disarm=lambda: rt.refuse_launch(-1))
        if got[0] == W.WS_OK:
            check(ref, got)
        else:
            assert got[0] == W.WS_ERR_CUDA
            lost += 1
    assert 0 < lost < n  # plain launches have no substitute, the fused ones have


@pytest.mark.parametrize("case", UPDATES)
def test_updates(case, tmp_path):
    need_gpu()
    child("refuse_updates", tmp_path, case, module="test_gpu_refused_launch")


@pytest.mark.parametrize("case", UPDATES)
def test_earlier_error_is_not_the_updates(case):
    # an error that another call of the thread left in the runtime
    need_gpu()
    rt = ctypes.CDLL("libcudart.so.13")

    def leave_error():
        assert rt.cudaSetDevice(1 << 20) != 0 and rt.cudaPeekAtLastError() != 0
    ref = update(*case)
    got = update(*case, arm=leave_error, disarm=rt.cudaGetLastError)
    assert ref[0] == got[0] == W.WS_OK
    for x, y in zip(ref[1] + ref[2], got[1] + got[2]):
        assert np.array_equal(x, y)


def refuse_rollouts(rt):
    """Every launch of a roll-out (captured) and of a step (direct), on the FP32 paths and the BF16 path's layers."""
    for path in (W.WS_PATH_BATCHED_FP32, W.WS_PATH_PLAIN_FP32, W.WS_PATH_BATCHED_BF16):
        for env, n in ((W.WS_ENV_ECONOMY, 5), (W.WS_ENV_LANDSCAPE, 20), (W.WS_ENV_CONTROL, 20)):
            for call in (lambda r: W.ws_rollout(r.ctx, 2), lambda r: W.ws_step(r.ctx)):
                def run(i):
                    r = context(env, 64, n, 4, 8, path=path)
                    rt.refuse_launch(i)
                    st, seen = call(r), rt.launches_seen()
                    rt.refuse_launch(-1)
                    again = W.ws_step(r.ctx)
                    r.close()
                    return seen, st, again
                seen, st, again = run(-1)
                assert st == again == W.WS_OK
                for i in range(seen):
                    assert run(i)[1:] == (W.WS_ERR_CUDA, W.WS_ERR_CUDA), (path, env, i)


def refuse_post_passes(rt):
    """Every launch of the forces, the returns and a reset, on each path (BF16: the tensor-core force)."""
    for path, h in ((W.WS_PATH_PLAIN_FP32, 64), (W.WS_PATH_BATCHED_FP32, 64), (W.WS_PATH_BATCHED_BF16, 256)):
        for call in (lambda r: W.ws_forces(r.ctx, 2), lambda r: W.ws_returns(r.ctx, 2), lambda r: W.ws_reset(r.ctx, 7)):
            def run(i):
                r = context(W.WS_ENV_LANDSCAPE, h, 20, 4, 8, W.WS_FLAG_FORCE, path)
                r.rollout(2)
                rt.refuse_launch(i)
                st, seen = call(r), rt.launches_seen()
                rt.refuse_launch(-1)
                r.close()
                return seen, st
            seen, st = run(-1)
            assert st == W.WS_OK and seen > 0
            for i in range(seen):
                assert run(i)[1] == W.WS_ERR_CUDA, (path, i)


def refuse_creation(rt):
    """Every launch of ws_create and of ws_load (parameters), on each path."""
    shapes = [(W.WS_ENV_CONTROL, 64), (W.WS_ENV_ACROBOT, 64), (W.WS_ENV_ECONOMY, 128), (W.WS_ENV_ECONOMY, 64),
              (W.WS_ENV_LANDSCAPE, 256), (W.WS_ENV_LANDSCAPE, 64)]
    for path in (W.WS_PATH_PLAIN_FP32, W.WS_PATH_BATCHED_FP32, W.WS_PATH_BATCHED_BF16):
        for env, h in shapes:
            flags = W.WS_FLAG_TRAIN | (W.WS_FLAG_FORCE if env == W.WS_ENV_LANDSCAPE else 0)
            kw = dict(dim=8, n_gauss=64) if env == W.WS_ENV_LANDSCAPE else {}

            def create(i):
                rt.refuse_launch(i)
                try:
                    r, st = W.Rollout(env, path, 5, 4, 9, h, h, flags=flags, **kw), W.WS_OK
                except W.WarpSciError as e:
                    r, st = None, e.status
                seen = rt.launches_seen()
                rt.refuse_launch(-1)
                return r, st, seen
            r, st, seen = create(-1)
            assert st == W.WS_OK and seen > 0
            n = sum(a * b + b for a, b in ((r.obs_dim(), h), (h, h), (h, r.n_out())))
            n += sum(a * b + b for a, b in ((16, h), (h, h), (h, 10))) if env == W.WS_ENV_ECONOMY else 0
            params = np.zeros(n, np.float32)

            def load(r, i):
                rt.refuse_launch(i)
                st = W.ws_load(r.ctx, W.WS_F_PARAMS, params.ctypes.data, params.nbytes, 0, 2 ** 64 - 1)
                got = st, rt.launches_seen()
                rt.refuse_launch(-1)
                r.close()
                return got
            for i in range(seen):
                assert create(i)[:2] == (None, W.WS_ERR_CUDA), (path, env, h, i)
            st, seen = load(r, -1)
            assert st == W.WS_OK
            for i in range(seen):
                assert load(create(-1)[0], i)[0] == W.WS_ERR_CUDA, (path, env, h, i)


def refuse_forward(rt):
    import torch
    x, w, y = (torch.zeros(4096, device="cuda") for _ in range(3))

    def call(out):
        return W.ws_policy_forward_noalloc(x.data_ptr(), 3, w.data_ptr(), 4, 16, 16, 2, out.data_ptr(), 0)
    for out in (y, x):  # one launch; over the input, layer by layer
        rt.refuse_launch(-1)
        assert call(out) == W.WS_OK
        for i in range(rt.launches_seen()):
            rt.refuse_launch(i)
            assert call(out) == W.WS_ERR_CUDA
        rt.refuse_launch(-1)
        assert call(out) == W.WS_OK


@pytest.mark.parametrize("what", ["refuse_creation", "refuse_rollouts", "refuse_post_passes", "refuse_forward"])
def test_calls_without_a_substitute(what, tmp_path):
    need_gpu()
    child(what, tmp_path, module="test_gpu_refused_launch")


@pytest.mark.parametrize("path", [W.WS_PATH_PLAIN_FP32, W.WS_PATH_BATCHED_FP32, W.WS_PATH_BATCHED_BF16])
def test_earlier_error_is_not_the_rollouts(path):
    need_gpu()
    rt = ctypes.CDLL("libcudart.so.13")
    for env in (W.WS_ENV_ECONOMY, W.WS_ENV_LANDSCAPE, W.WS_ENV_CONTROL):
        r = context(env, 64, 5, 4, 8, path=path)
        for call in (lambda: W.ws_step(r.ctx), lambda: W.ws_rollout(r.ctx, 2)):
            assert rt.cudaSetDevice(1 << 20) != 0 and rt.cudaPeekAtLastError() != 0
            assert call() == W.WS_OK
        r.sync()
        r.close()
    rt.cudaGetLastError()
