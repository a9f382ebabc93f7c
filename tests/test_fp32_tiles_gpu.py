"""The fp32 kernels' tile shapes at their edges: row tiles of 8 to 128 rows, two and four key
groups, groups without a key, feature counts between the column blocks."""
import numpy as np
import pytest

from gpu_helpers import assert_close, lse_bound, rel_err, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402
from paper_2606_07713_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.lib()


SHAPES = [
    (1, 1, 1, 64, 4, 4),          # one row; the second key group has no key
    (1, 2, 7, 65, 64, 64),        # the second group has one key
    (1, 3, 9, 257, 64, 36),       # four groups, the last step has one key
    (1, 5, 33, 130, 20, 8),       # four groups, two of them without a key
    (2, 9, 130, 300, 60, 100),    # columns past d_v in the last 32-column block
    (1, 20, 300, 129, 32, 96),    # 16-row tiles
    (1, 16, 65, 513, 64, 64),     # one row in the last tile, one key in the last step
    (4, 40, 129, 90, 64, 64),     # 128-row tiles, two groups
    (1, 9, 520, 193, 128, 128),   # two groups: four do not fit with d = 128
    (2, 16, 515, 70, 128, 32),    # N_q past the four-group range
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_fp32_tile_edges(oracle, shape):
    """Forward and log-sum-exp within the fp32 bound, gradients within twice that (dP - D cancels),
    and one (b, h) slice alone bit-equal to the same slice of the whole call."""
    cfg = I.custom_config(*shape, dtype="fp32", seed=sum(shape) + 3)
    x = I.make_inputs(cfg)
    g, _ = I.make_grad_output(cfg)
    q, k, v = to_device(x)
    do = torch.from_numpy(np.ascontiguousarray(g)).to("cuda:0")
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    grads = pkg.attn_bwd(q, k, v, o, lse, do, x.scale)
    ref, lref = oracle.attn_lse(x.q, x.k, x.v, x.scale)
    assert_close(o.cpu().numpy(), ref, "fp32", str(shape))
    assert np.all(np.abs(lse.double().cpu().numpy() - lref) <= lse_bound(x, lref))
    for name, a, b in zip(("dQ", "dK", "dV"), grads, oracle.attn_bwd(x.q, x.k, x.v, g, x.scale)):
        a = a.cpu().numpy()
        assert np.all(np.isfinite(a)), name
        err = np.max(np.abs(a)) if np.max(np.abs(b)) == 0.0 else rel_err(a, b)
        assert err <= 2e-5, f"{shape} {name}: {err:.3e}"
    b, h = shape[0] - 1, shape[1] - 1
    one = [t[b:b + 1, h:h + 1].contiguous() for t in (q, k, v, o, lse, do)]
    o1, lse1 = pkg.attn_fwd_lse(*one[:3], x.scale)
    assert torch.equal(o1[0, 0], o[b, h]) and torch.equal(lse1[0, 0], lse[b, h])
    for a, whole in zip(pkg.attn_bwd(*one, x.scale), grads):
        assert torch.equal(a[0, 0], whole[b, h])


@pytest.mark.parametrize("masked", [(1, 3), (0, 2, 4), (1, 2, 3), (0, 1)])
@pytest.mark.parametrize("nq", [9, 520])
def test_tiles_of_masked_keys(oracle, nq, masked):
    """Keys whose score is -inf (first feature: 1 in Q, -inf in K) have no part in the result, also
    where a key group (64 keys of each step) has no other keys, or none in its first step."""
    x = I.make_inputs(I.custom_config(1, 2, nq, 370, 64, 64, dtype="fp32", seed=nq + len(masked)))
    keep = [i for i in range(370) if i // 64 not in masked]
    x.q[..., 0] = 1.0
    x.k[..., 0] = 0.0
    q, k, v = to_device(x)
    km = torch.full_like(k[..., 0], float("-inf"))
    km[..., keep] = 0.0
    k[..., 0] = km
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    ref, lref = oracle.attn_lse(x.q, x.k[:, :, keep].copy(), x.v[:, :, keep].copy(), x.scale)
    assert_close(o.cpu().numpy(), ref, "fp32", f"{nq} {masked}")
    assert np.all(np.abs(lse.double().cpu().numpy() - lref) <= lse_bound(x, lref))
