"""The sizer's kernels at sizes around their tiles (32-vertex chunks, 64-row
products, 8 warps to a block), and large copies to the host at the edges of
their staging buffers."""
import numpy as np
import pytest

from oracle import sizer_ref as R
from paper_2210_16998_gb300 import cfggen as G
from paper_2210_16998_gb300 import tpg

from .test_gpu_sizer import load_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains", [(1,), (10,), (1, 9), (21,), (21, 10), (32, 31, 1), (85,) * 10])
def test_gradient_and_totals(chains):
    cfgs = [G.diamond_chain(k) for k in chains]
    X, A = R.batch_inputs(cfgs)
    h, N = load_batch(cfgs)
    assert N == sum(3 * k + 1 for k in chains)
    with h, tpg.tpg_sizer_create(seed=5) as z:
        if max(chains) <= 21:  # (labels need an exact count)
            tpg.tpg_sizer_add_batch(z, h)
            T = tpg.tpg_sizer_batch_targets(z, 0, N).astype(np.float64)
        p = np.random.default_rng(len(chains)).normal(0.0, 0.15, R.NPARAM).astype(np.float32)
        tpg.tpg_sizer_set_params(z, p)
        pred, totals = tpg.tpg_sizer_predict(z, h, N)
        # the network rounds to bf16 (2^-9) in about eight places on a path
        ref = R.forward(p.astype(np.float64), X, A, bf=True)
        ref = ref[0] if isinstance(ref, tuple) else ref
        np.testing.assert_allclose(pred, ref, rtol=8 * 2.0 ** -8, atol=8 * 2.0 ** -8 * np.abs(ref).max())
        exact = np.expm1(np.maximum(pred.astype(np.float64), 0.0)).sum(0)
        np.testing.assert_allclose(totals, exact, rtol=1e-12)
        if max(chains) > 21:
            return
        loss, g = tpg.tpg_sizer_loss_grad(z, 0)
        rl, rg = R.loss_grad(p.astype(np.float64), X, A, T, bf=True)
        assert abs(loss - rl) <= 8 * 2.0 ** -8 * rl
        assert np.linalg.norm(g - rg) <= 16 * 2.0 ** -8 * np.linalg.norm(rg)


@pytest.mark.parametrize("extra", [-1, 0, 1, 1023, 1024, 1025])
@pytest.mark.parametrize("dtype", ["int32", "int64"])
def test_large_copies_to_the_host(monkeypatch, extra, dtype):
    import torch

    monkeypatch.setattr(tpg, "_STAGE_BYTES", 8192)
    n = 2 * 8192 // np.dtype(dtype).itemsize + extra
    t = torch.arange(n, dtype=getattr(torch, dtype), device="cuda") * 3 - 7
    got = tpg._to_host(t)
    assert got.dtype == np.dtype(dtype)
    np.testing.assert_array_equal(got, np.arange(n, dtype=dtype) * 3 - 7)
