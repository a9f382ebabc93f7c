"""The fused backward kernel at its edges, on grids that run it: attn_bwd(fused=True) takes
moa_attn_bwd's kernels where those are estimated to take less, which is most small calls, so every case
asks moa_attn_bwd_fused_plan first.  Tolerance: that of the existing parity tests of the gradients."""
import numpy as np
import pytest

from gpu_helpers import BF16_TOL, rel_err
from test_bwd_fused_gpu import grads

import paper_2606_07713_gb300 as pkg
from paper_2606_07713_gb300 import _lib
from paper_2606_07713_gb300 import inputs as I

torch = pytest.importorskip("torch")


def need_fused(*shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert pkg.moa_attn_bwd_fused_plan(*shape[:4], 0) == (0, 1), f"{shape} does not run the fused kernel"


# ragged remainders of keys and queries, one key, one row past a block, one slice, many
SHAPES = [(4, 37, 300, 3), (4, 37, 257, 1), (4, 35, 129, 300), (4, 35, 300, 129), (2, 37, 1000, 129),
          (4, 12, 260, 300), (2, 1, 513, 2048)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_fused_parity(oracle, shape):
    need_fused(*shape)
    x = I.make_inputs(I.custom_config(*shape, 64, 64, dtype="bf16", seed=sum(shape)))
    g, gb = I.make_grad_output(x.cfg)
    got = [t.float().cpu().numpy() for t in grads(x, gb, True)]
    for name, a, b in zip(("dQ", "dK", "dV"), got, oracle.attn_bwd(x.q, x.k, x.v, g, x.scale)):
        assert np.all(np.isfinite(a)), name
        err = np.max(np.abs(a)) if np.max(np.abs(b)) == 0.0 else rel_err(a, b)
        assert err <= (1e-3 if np.max(np.abs(b)) == 0.0 else BF16_TOL), f"{shape} {name}: {err:.3e}"


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [-0.3, 2.0 / 8, 0.0])
def test_fused_other_scales(oracle, scale):
    need_fused(4, 6, 260, 700)
    x = I.make_inputs(I.custom_config(4, 6, 260, 700, 64, 64, dtype="bf16", seed=77))
    g, gb = I.make_grad_output(x.cfg)
    got = [t.float().cpu().numpy() for t in grads(x, gb, True, scale=scale)]
    for name, a, b in zip(("dQ", "dK", "dV"), got, oracle.attn_bwd(x.q, x.k, x.v, g, scale)):
        assert np.all(np.isfinite(a)), name
        if np.max(np.abs(b)) == 0.0:
            assert np.max(np.abs(a)) <= 1e-3, name
        else:
            assert rel_err(a, b) <= BF16_TOL, f"{scale} {name}: {rel_err(a, b):.3e}"


@pytest.mark.gpu
def test_fused_dk_dv_reproducible_and_sum_rules():
    """dK and dV bit for bit from run to run, dQ up to the order of its additions; the value gradients sum
    to the column sums of dO, and <dQ, Q> = <dK, K> per head."""
    need_fused(4, 8, 1024, 1024)
    x = I.make_inputs(I.custom_config(4, 8, 1024, 1024, 64, 64, dtype="bf16", seed=5))
    g, gb = I.make_grad_output(x.cfg)
    a, b = grads(x, gb, True), grads(x, gb, True)
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert (a[0].float() - b[0].float()).abs().max().item() <= 1e-2 * a[0].float().abs().max().item()
    dq, dk, dv = (t.double().cpu().numpy() for t in a)
    colsum = g.astype(np.float64).sum(axis=2)
    assert np.max(np.abs(dv.sum(axis=2) - colsum)) <= 2e-2 * np.max(np.abs(colsum)) + 1e-2
    lhs = np.sum(dq * x.q.astype(np.float64), axis=(2, 3))
    rhs = np.sum(dk * x.k.astype(np.float64), axis=(2, 3))
    assert np.max(np.abs(lhs - rhs)) <= 3e-2 * np.max(np.abs(rhs)) + 1e-2


def test_plan_without_a_gpu():
    """The choice on 152 SMs: the listed cases of this file and the training size run the fused kernel,
    one block pair and one long head do not; bad sizes are refused."""
    from paper_2606_07713_gb300 import build
    build.build()
    for shape in SHAPES + [(4, 6, 260, 700), (4, 8, 1024, 1024), (4, 16, 2048, 2048)]:
        assert pkg.moa_attn_bwd_fused_plan(*shape, 152) == (0, 1), shape
    for shape in [(1, 1, 92, 92), (6, 8, 661, 84), (3, 5, 500, 1500), (1, 1, 8000, 8000)]:
        assert pkg.moa_attn_bwd_fused_plan(*shape, 152) == (0, 0), shape
    for shape in [(0, 1, 1, 1), (1, 1, -1, 1), (1 << 31, 1 << 31, 1 << 31, 1)]:
        assert pkg.moa_attn_bwd_fused_plan(*shape, 152)[0] == _lib.MOA_ERR_INVALID_ARG
