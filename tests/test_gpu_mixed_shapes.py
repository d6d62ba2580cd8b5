"""Contexts of different shapes that share kernels: none changes what another one's launches need."""
import threading

import numpy as np
import pytest

from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import need_gpu
from tests.refuse_launch import child

pytestmark = pytest.mark.gpu


def train(dim, h, torch, times=1):
    """Parameters after updates of a landscape policy, on a stream of its own."""
    with torch.cuda.stream(torch.cuda.Stream()):
        r = W.Rollout(W.WS_ENV_LANDSCAPE, W.WS_PATH_BATCHED_FP32, 130, 2, 9, h, h, dim=dim, n_gauss=64, param_seed=5,
                      flags=W.WS_FLAG_TRAIN)
        r.reset(6)
        r.rollout(2)
        for _ in range(times):
            r.a2c_update(2, 0.1, 0.5, 0.01)
        n = dim * h + h + h * h + h + h * 2 * dim + 2 * dim
        p = r.fetch_raw(W.WS_F_PARAMS, 4 * n).copy()
        r.close()
    return p


def update_limits(rt):
    import torch
    for h in (64, 128, 256):
        for dim in (1, 4, 5, 16, 17, 24):
            train(dim, h, torch)
    assert rt.limits_changed() == 0


def test_updates_set_one_limit(tmp_path):
    # the limit of shared memory is the kernel's, not the context's: a lower one set by another thread between this
    # thread's setting and its launch would have the launch refused
    need_gpu()
    child("update_limits", tmp_path, module="test_gpu_mixed_shapes")


def test_updates_in_threads():
    torch = need_gpu()
    dims = (17, 24, 20, 23)
    ref = [train(d, 64, torch, 40) for d in dims]
    got = [None] * len(dims)

    def work(i):
        got[i] = train(dims[i], 64, torch, 40)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(dims))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(ref, got):
        assert b is not None and np.array_equal(a, b)


def test_landscapes_of_different_sizes():
    # a small BF16 landscape created after a large one
    need_gpu()
    make = lambda m: W.Rollout(W.WS_ENV_LANDSCAPE, W.WS_PATH_BATCHED_BF16, 200, 4, 3, 256, 256, dim=24, n_gauss=m)  # noqa: E731
    large = make(4096)
    want = large.fetch_raw(W.WS_F_STATE, 200 * (24 + 2) * 4)
    small = make(64)
    large.reset(large.cfg.param_seed)
    large.sync()
    assert np.array_equal(large.fetch_raw(W.WS_F_STATE, 200 * (24 + 2) * 4), want)
    small.close()
    large.close()
