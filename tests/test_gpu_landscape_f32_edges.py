"""FP32 landscape energy and force against the FP64 oracle at the edges of their tiles: coordinate counts on both sides
of each register width, odd Gaussian counts (the force kernel takes two at a time, 128 per tile in four quarters; the
energy kernel eight at a time, 64 per tile in eight chunks), states near centres.  Tolerances as the larger shapes'
(test_gpu_landscape.py, test_gpu_force.py)."""
import numpy as np
import pytest

import oracle
from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import TOL_F32, need_gpu
from tests.test_gpu_force import TOL_FORCE_F32, env_params, force_scale
from tests.ws_helpers import pack_landscape_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [W.WS_PATH_PLAIN_FP32, W.WS_PATH_BATCHED_FP32])
@pytest.mark.parametrize("dim,gauss", [(1, 1), (1, 129), (5, 1), (5, 33), (5, 70), (8, 129), (8, 333), (9, 7), (16, 33),
                                       (16, 333), (24, 1), (24, 513), (25, 129), (32, 33), (32, 333), (33, 64), (33, 65),
                                       (64, 1), (64, 130)])
def test_energy_and_force(path, dim, gauss):
    need_gpu()
    n = 67  # past one tile of 64 rows
    g = np.random.default_rng(dim * 1000 + gauss)
    r = W.Rollout(W.WS_ENV_LANDSCAPE, path, n, 2, 1000, 16, 16, dim=dim, n_gauss=gauss, param_seed=7, noise_sigma=0.0,
                  flags=W.WS_FLAG_FORCE | W.WS_FLAG_BOUNDS_CHECK)
    c, w, a = env_params(r, gauss, dim)
    x0 = (c[g.integers(0, gauss, n)] + g.normal(0, 0.3, (n, dim))).astype(np.float32)
    r.load_raw(W.WS_F_STATE, pack_landscape_state(x0, np.zeros(n), np.zeros(n)), k=0)
    r.rollout(2)
    r.forces(2)
    r.sync()
    obs, act, en, force = (r.fetch(f, 0, 2) for f in (W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_ENERGY, W.WS_F_FORCE))
    r.close()
    assert np.abs(en).max() > 1e-3
    for t in range(2):
        for e in range(n):
            y = (obs[t][:, e] + act[t][:, e]).astype(np.float32).astype(np.float64)
            sc = oracle.landscape_energy_scale(c, w, a, y)
            assert abs(en[t][e] - oracle.landscape_energy(c, w, a, y)) <= TOL_F32 * max(sc, 1e-3) + 1e-7, (t, e)
            ref, fs = -oracle.landscape_grad(c, w, a, y), np.maximum(force_scale(c, w, a, y), 1e-3)
            assert (np.abs(force[t][:, e] - ref) / fs).max() <= TOL_FORCE_F32, (t, e)
