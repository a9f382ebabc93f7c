"""Backward at ragged lengths: the rows that complete the last tile of keys or queries weigh nothing,
whatever the real rows hold.  Tolerances are those of the parity tests (bf16 2e-2, fp32 2e-5 of the
largest gradient): the inputs below change no rounding, only which padded products would overflow."""
import numpy as np
import pytest

from gpu_helpers import BF16_TOL, bf16_tensor_from_f32, rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402
from paper_2606_07713_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.lib()


def bf16(a):
    return I.bf16_bits_to_f32(I.f32_to_bf16_bits(np.asarray(a, dtype=np.float32)))


def device(a, dtype):
    if dtype == "bf16":
        return bf16_tensor_from_f32(a)
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def gradients(q, k, v, g, scale, dtype, fused):
    t = [device(a, dtype) for a in (q, k, v, g)]
    o, lse = pkg.attn_fwd_lse(*t[:3], scale)
    out = pkg.attn_bwd(*t[:3], o, lse, t[3], scale, fused=fused)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    return lse, [x.float().cpu().numpy() for x in out]


@pytest.mark.parametrize("grid", [(2, 9, 100, 64, 64, "fp32", False), (1, 200, 300, 32, 96, "fp32", False)],
                         ids=str)
def test_masked_keys_with_ragged_queries(oracle, grid):
    """Keys that score -inf (first feature: 1 in Q, -inf in K) have zero dK and dV: the zeros that
    complete the last query tile make 0 * -inf of their scores, which must not count.  dQ's first
    feature is 0 * -inf by definition and is left out."""
    bh, nq, nk, dk, dv, dtype, fused = grid
    r = np.random.default_rng(sum(grid[:5]))
    rnd = bf16 if dtype == "bf16" else np.float32
    q, k, v, g = (rnd(r.standard_normal((1, bh, n, d))) for n, d in ((nq, dk), (nk, dk), (nk, dv), (nq, dv)))
    masked = np.arange(nk) % 3 == 1
    q[..., 0] = 1.0
    k[..., 0] = np.where(masked, -np.inf, 0.0)
    scale = dk ** -0.5
    _, (dq, dk_, dv_) = gradients(q, k, v, g, scale, dtype, fused)
    assert np.all(dk_[:, :, masked] == 0.0) and np.all(dv_[:, :, masked] == 0.0)
    keep = ~masked
    tol = BF16_TOL if dtype == "bf16" else 2e-5
    for h in (0, bh - 1):
        s = (slice(0, 1), slice(h, h + 1))
        ref = oracle.attn_bwd(q[s], k[s][:, :, keep].copy(), v[s][:, :, keep].copy(), g[s], scale)
        got = (dq[s][..., 1:], dk_[s][:, :, keep], dv_[s][:, :, keep])
        for name, a, b in zip(("dQ", "dK", "dV"), got, (ref[0][..., 1:], ref[1], ref[2])):
            assert np.all(np.isfinite(a)), name
            assert rel_err(a, b) <= tol, f"{name} of slice {h}: {rel_err(a, b):.3e}"
