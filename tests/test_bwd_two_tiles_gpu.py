"""The two-tile dQ kernel, which large grids take: its rows are the one-tile kernel's bit for bit, at
the edges of its 256-row blocks, and the gradients hold against the oracle."""
import numpy as np
import pytest

from gpu_helpers import BF16_TOL, rel_err, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402
from paper_2606_07713_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.lib()


@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (128, 64), (64, 128)])
@pytest.mark.parametrize("nq,nk", [(512, 129), (385, 300), (513, 128)])
def test_two_tile_dq_matches_one_tile_and_oracle(oracle, nq, nk, dk, dv):
    """160 slices fill the GPU (two tiles per CTA); a slice alone does not (one tile).  Row counts:
    whole blocks, a second tile with one row, a block whose second tile is empty."""
    cfg = I.custom_config(10, 16, nq, nk, dk, dv, dtype="bf16", seed=nq + nk + dk)
    x = I.make_inputs(cfg)
    g, gb = I.make_grad_output(cfg)
    q, k, v = to_device(x)
    do = torch.from_numpy(np.ascontiguousarray(gb).view(np.int16)).view(torch.bfloat16).to("cuda:0")
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    grads = pkg.attn_bwd(q, k, v, o, lse, do, x.scale)
    for b, h in ((0, 0), (9, 15)):
        one = pkg.attn_bwd(*(t[b:b + 1, h:h + 1].contiguous() for t in (q, k, v, o, lse, do)), x.scale)
        for name, a, whole in zip(("dQ", "dK", "dV"), one, grads):
            assert torch.equal(a[0, 0], whole[b, h]), f"{name} of slice {b},{h}"
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    s = (slice(9, 10), slice(15, 16))
    ref = oracle.attn_bwd(x.q[s], x.k[s], x.v[s], g[s], x.scale)
    for name, a, b in zip(("dQ", "dK", "dV"), grads, ref):
        err = rel_err(a[s].float().cpu().numpy(), b)
        assert err <= BF16_TOL, f"{name}: {err:.3e}"
