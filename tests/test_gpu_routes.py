"""Calls that reach a kernel or a branch by a rule on their sizes, on both
sides of the rule: the tensor path's pair tiles, its class shift, order 2's
automatic path, thresholds and whole score tables counted on the tensor
cores, merges of small and large pools, batches with studies searched alone,
and the fused training kernels."""
from __future__ import annotations

import itertools
import math

import numpy as np
import pytest

from oracle import mlp as M
from oracle import oracle as O
from tests.helpers import F32_RTOL, check_topn, random_data
from tests.test_gpu_learn import _bf16, _grad_magnitudes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def epi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_02460_gb300 import epi as E
    E.load()
    return E


@pytest.fixture(scope="module")
def ctx(epi):
    return epi.Context(0)


# fused training kernels: rows around a tile and beyond one tile a block
# (512 x 32), inputs and hidden units at the rule's edges; (33 inputs, 288
# hidden units: the separate kernels).  Bounds as for the gradients of other
# shapes: differing terms of BF16 storage, FP32 sums, masks near zero.
@pytest.mark.parametrize("rows,n_in,hidden", [(1, 1, 32), (31, 5, 32), (33, 32, 96), (100, 33, 64), (65, 30, 288),
                                              (257, 30, 256), (16417, 7, 64)])
def test_fused_gradients(epi, ctx, rows, n_in, hidden):
    import torch
    rng = np.random.default_rng(rows)
    net = epi.MLP(ctx, n_in, hidden, seed=rows)
    theta = net.params().astype(np.float64)
    X = rng.standard_normal((rows, n_in)).astype(np.float32)
    y, (_, _, _, _, H2, _, W3) = M.forward(theta, X, n_in, hidden, rnd=_bf16)
    scale = np.abs(H2) @ np.abs(W3) + 1.0
    t = (y + 4.0 * scale * np.where(np.arange(rows) % 2 == 0, 1.0, -1.0)).astype(np.float32)
    g, loss = net.gradients(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda())
    g2, loss2 = net.gradients(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda())
    assert (g == g2).all()
    want = M.gradients(theta, X, t, n_in, hidden, rnd=_bf16, rnd_dz=_bf16)
    S, L, A = _grad_magnitudes(theta, X, t, n_in, hidden, _bf16)
    err = np.abs(g.astype(np.float64) - want)
    assert (err <= 2.0 ** -6 * L + 2.0 ** -12 * S + A + 1e-30).all()
    assert abs(loss - M.loss(theta, X, t, n_in, hidden, rnd=_bf16)) <= 1e-4 * abs(loss) + 1e-7
    net.close()
