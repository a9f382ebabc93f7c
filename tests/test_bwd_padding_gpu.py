"""Backward at ragged lengths: the rows that complete the last tile of keys or queries weigh nothing,
whatever the real rows hold."""
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


# (slices, N_q, N_k, d_k, d_v, fused): one- and two-tile dQ CTAs, the fused kernel
GRIDS = [(2, 200, 129, 64, 64, False), (2, 200, 300, 128, 64, False), (160, 385, 129, 128, 128, False),
         (160, 385, 300, 64, 128, False), (148, 300, 129, 64, 64, True), (2, 300, 1000, 64, 64, True)]


@pytest.mark.parametrize("grid", GRIDS, ids=str)
def test_strongly_negative_scores(grid):
    """Q near +c and K near -c: every score is near -170, so the rows' log-sum-exp is below -88, where
    the weight exp(0 - LSE) of a key that does not exist overflows.  The gradients are those of the same
    call with its last block filled up by keys of weight exp(-320) = 0, bit for bit; the fused kernel's
    dQ up to the order of its additions."""
    bh, nq, nk, dk, dv, fused = grid
    r = np.random.default_rng(sum(grid[:5]))
    c = 4.5 if dk == 64 else 3.75
    q = bf16(c + 0.25 * r.standard_normal((1, bh, nq, dk)))
    k = bf16(-c + r.standard_normal((1, bh, nk, dk)))
    v, g = (bf16(r.standard_normal((1, bh, n, dv))) for n in (nk, nq))
    scale = dk ** -0.5
    fill = -nk % 128
    q, k, v, g = (device(a, "bf16") for a in (q, k, v, g))
    o, lse = pkg.attn_fwd_lse(q, k, v, scale)
    assert lse.max().item() < -100.0
    kf = torch.cat([k, torch.full_like(k[:, :, :1], -3 * c).expand(-1, -1, fill, -1)], 2)
    vf = torch.cat([v, torch.ones_like(v[:, :, :1]).expand(-1, -1, fill, -1)], 2)
    got = pkg.attn_bwd(q, k, v, o, lse, g, scale, fused=fused)
    want = pkg.attn_bwd(q, kf, vf, o, lse, g, scale, fused=fused)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    assert all(torch.all(torch.isfinite(t)) for t in got)
    if fused:
        dq_err = (got[0].float() - want[0].float()).abs().max().item()
        assert dq_err <= 1e-2 * want[0].float().abs().max().item()
    else:
        assert torch.equal(got[0], want[0])
    assert torch.equal(got[1], want[1][:, :, :nk]) and torch.equal(got[2], want[2][:, :, :nk])


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
