"""The one-launch FP32 policy forward, the register-tiled landscape energy and the force kernel.

Batched FP32 roll-outs of the economy and the landscape against the plain path's layer-by-layer kernels, byte for
byte (same arithmetic per output; the plain path is compared with the FP64 oracle elsewhere): widths on both sides
of each tile, coordinates that are and are not multiples of four, env counts at the edges of the row tiles.
ws_policy_forward_noalloc against the FP64 oracle at the tiles' edges, and with the output over the input."""
import numpy as np
import pytest

import oracle
from paper_2408_00930_gb300 import inputs
from paper_2408_00930_gb300 import warpsci as W
from tests.gpu_common import TOL_F32, need_gpu

pytestmark = pytest.mark.gpu


def _records(env, path, n, T, h0, h1, dim, gauss, agents):
    kw = dict(dim=dim, n_gauss=gauss) if env == W.WS_ENV_LANDSCAPE else dict(agents_per_env=agents)
    r = W.Rollout(env, path, n, T, 4, h0, h1, param_seed=3,
                  flags=W.WS_FLAG_DEBUG_LOGITS | W.WS_FLAG_BOUNDS_CHECK, **kw)
    r.reset(11)
    r.rollout(T)
    r.sync()
    fields = [W.WS_F_OBS, W.WS_F_ACTION, W.WS_F_LOGP, W.WS_F_REWARD, W.WS_F_DONE, W.WS_F_POLICY_OUT]
    fields.append(W.WS_F_ENERGY if env == W.WS_ENV_LANDSCAPE else W.WS_F_WEALTH)
    out = [r.fetch(f, 0, T) for f in fields]
    r.close()
    return out


@pytest.mark.parametrize("env,n,h0,h1,dim,gauss", [
    (W.WS_ENV_LANDSCAPE, 1, 64, 64, 1, 1), (W.WS_ENV_LANDSCAPE, 257, 100, 37, 5, 70),
    (W.WS_ENV_LANDSCAPE, 1300, 64, 64, 24, 513), (W.WS_ENV_LANDSCAPE, 255, 256, 256, 24, 65),
    (W.WS_ENV_LANDSCAPE, 3000, 256, 200, 33, 64), (W.WS_ENV_LANDSCAPE, 5100, 129, 256, 64, 130),
    (W.WS_ENV_ECONOMY, 3, 128, 128, 0, 0), (W.WS_ENV_ECONOMY, 40, 100, 66, 0, 0),
    (W.WS_ENV_ECONOMY, 300, 128, 128, 0, 0)])
def test_batched_fp32_equals_plain(env, n, h0, h1, dim, gauss):
    agents = np.random.default_rng(4).integers(2, 300, n) if env == W.WS_ENV_ECONOMY else None
    a = _records(env, W.WS_PATH_PLAIN_FP32, n, 6, h0, h1, dim, gauss, agents)
    b = _records(env, W.WS_PATH_BATCHED_FP32, n, 6, h0, h1, dim, gauss, agents)
    for i, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x.view(np.uint8), y.view(np.uint8)), i


@pytest.mark.parametrize("rows,widths", [
    (1, (1, 1, 1, 1)), (7, (3, 5, 2, 128)), (300, (16, 128, 128, 20)), (1217, (64, 64, 33, 48)),
    (2433, (6, 256, 255, 3)), (4865, (24, 250, 256, 49)), (31000, (4, 66, 66, 2))])
def test_noalloc_forward_edges(rows, widths):
    torch = need_gpu()
    g = inputs.rng(rows)
    params = inputs.policy_params(g, list(widths), scale=2.0)
    x = g.uniform(-1, 1, (rows, widths[0])).astype(np.float32)
    ref = oracle.mlp_forward(list(widths), params, x.astype(np.float64))
    p = torch.from_numpy(params).cuda()
    for over in (False, True):  # the output over the input: refused by no check, served layer by layer
        buf = torch.zeros(rows * max(widths[0], widths[3]), device="cuda")
        obs = buf[:rows * widths[0]]
        obs.copy_(torch.from_numpy(x).reshape(-1))
        out = buf if over else torch.full((rows * widths[3],), float("nan"), device="cuda")
        st = W.ws_policy_forward_noalloc(obs.data_ptr(), rows, p.data_ptr(), *widths, out.data_ptr(),
                                         torch.cuda.current_stream().cuda_stream)
        assert st == W.WS_OK
        got = out[:rows * widths[3]].cpu().numpy().reshape(rows, widths[3])
        err = np.abs(got - ref) / np.maximum(np.abs(ref).max(axis=1, keepdims=True), 1.0)
        assert err.max() <= TOL_F32


@pytest.mark.parametrize("rows,widths", [
    (1, (24, 128, 128, 48)), (9, (1, 65, 128, 33)), (1215, (16, 128, 37, 17)), (2432, (23, 100, 66, 32)),
    (2431, (4, 64, 64, 16)), (8, (24, 33, 64, 48))])
def test_noalloc_forward_few_rows(rows, widths):
    test_noalloc_forward_edges(rows, widths)


@pytest.mark.parametrize("rows,widths", [
    (9, (3, 33, 37, 5)), (300, (4, 61, 100, 20)), (9, (30, 33, 37, 60)), (9, (5, 250, 130, 3)),
    (4900, (4, 66, 66, 2)), (31000, (4, 61, 33, 2)), (9000, (7, 129, 250, 4))])
def test_infinite_inputs_match_the_layers(rows, widths):
    # a unit past the width sees inf * 0: it must stay out of the next layer, as in the layer-by-layer forward
    torch = need_gpu()
    g = inputs.rng(rows)
    p = torch.from_numpy(inputs.policy_params(g, list(widths), scale=2.0)).cuda()
    x = g.uniform(-1, 1, (rows, widths[0])).astype(np.float32)
    x[1, 0], x[rows - 1, widths[0] - 1] = np.inf, -np.inf
    x[rows // 2, 1] = np.nan
    got = []
    for over in (False, True):
        buf = torch.zeros(rows * max(widths[0], widths[3]), device="cuda")
        obs = buf[:rows * widths[0]]
        obs.copy_(torch.from_numpy(x).reshape(-1))
        out = buf if over else torch.empty(rows * widths[3], device="cuda")
        assert W.ws_policy_forward_noalloc(obs.data_ptr(), rows, p.data_ptr(), *widths, out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream) == W.WS_OK
        got.append(out[:rows * widths[3]].cpu().numpy().reshape(rows, widths[3]))
    assert np.isnan(got[1]).sum() == widths[3]  # the row with a NaN input, no other
    assert np.array_equal(got[0], got[1], equal_nan=True)
