"""The network's gradient at the edges of the kernel's sample tiles (32) and
with several tiles per block, against the fp64 oracle with the tolerances of
the gradient test in test_gpu_sched.py."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import mlp as M
from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import learned as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 300, 9728, 9729, 20011])
def test_gradient_tiles(n):
    torch = pytest.importorskip("torch")
    model = L.new_model(3)
    w = (model.w.cpu().numpy().view(np.uint16).astype(np.uint32) << 16).view(np.float32)
    rng = np.random.default_rng(n)
    X = rng.normal(1, 1, (n, 8)).astype(np.float32)
    T = rng.normal(2, 1, n).astype(np.float32)
    grad = torch.full((gpm.GPM_MLP_PARAMS,), 7.0, dtype=torch.float32, device="cuda")
    loss = torch.full((1,), 7.0, dtype=torch.float32, device="cuda")
    gpm.gpm_mlp_grad(model.w, torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), grad, loss)
    y, cache = M.forward(M.unflatten(w.astype(np.float64)), X)
    go = np.concatenate([M.backward(cache, T)[k].ravel() for k in M.ORDER])
    assert np.abs(grad.cpu().numpy() - go).max() <= 2e-3 * np.abs(go).max()
    assert abs(float(loss.item()) - M.loss(y, T)) <= 1e-4 * max(1.0, M.loss(y, T))
