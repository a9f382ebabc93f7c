"""Keys whose score is -inf (first feature: 1 in Q, -inf in K) have no part in the result, wherever
they stand: the first key blocks of a row, every key of a key group or of a key range.  A row without
any other key is 0/0: its output is NaN and its log-sum-exp -inf, as in any softmax."""
import numpy as np
import pytest

from gpu_helpers import assert_close, lse_bound, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402
from paper_2606_07713_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.lib()


def masked_inputs(shape, dtype, block, masked, value=float("-inf")):
    """Inputs whose key blocks `masked` (of `block` keys) score `value`; the oracle's inputs without them."""
    x = I.make_inputs(I.custom_config(*shape, dtype=dtype, seed=sum(shape) + len(masked)))
    keep = [i for i in range(shape[3]) if i // block not in masked]
    x.q[..., 0] = 1.0
    x.k[..., 0] = 0.0
    q, k, v = to_device(x)
    q[..., 0] = 1.0
    km = torch.full_like(k[..., 0], value)
    km[..., keep] = 0.0
    k[..., 0] = km
    return x, q, k, v, (x.q, x.k[:, :, keep].copy(), x.v[:, :, keep].copy())


def check_lse(scale, lse, ref, lref):
    # the bound of the finite keys: the masked ones add nothing to the sum of the scores' errors
    xf = type("X", (), {"q": ref[0], "k": ref[1], "scale": scale})
    assert np.all(np.abs(lse.double().cpu().numpy() - lref) <= lse_bound(xf, lref))


@pytest.mark.parametrize("nk,masked", [(192, (0, 1)), (256, (0, 1, 2)), (370, (0, 1, 4, 5)),
                                       (370, (0, 1, 2, 4, 5)), (500, (0, 1, 2, 3))])
@pytest.mark.parametrize("nq", [9, 520])
def test_fp32_key_groups_without_a_key(oracle, nq, nk, masked):
    """Blocks of 64 keys, as the key groups take them: two, three and four empty groups of four."""
    x, q, k, v, ref = masked_inputs((1, 2, nq, nk, 64, 64), "fp32", 64, masked)
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    oref, lref = oracle.attn_lse(*ref, x.scale)
    assert_close(o.cpu().numpy(), oref, "fp32", f"{nq} {nk} {masked}")
    check_lse(x.scale, lse, ref, lref)


DIMS = [(64, 64), (128, 128), (128, 64), (64, 128)]


@pytest.mark.parametrize("dk,dv", DIMS)
@pytest.mark.parametrize("nq", [50, 200])
@pytest.mark.parametrize("masked", [(0,), (0, 1, 2), (1, 2)])
def test_first_blocks(oracle, nq, dk, dv, masked):
    x, q, k, v, ref = masked_inputs((1, 2, nq, 500, dk, dv), "bf16", 128, masked)
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    oref, lref = oracle.attn_lse(*ref, x.scale)
    assert_close(o.float().cpu().numpy(), oref, "bf16", f"{nq} {dk},{dv} {masked}")
    check_lse(x.scale, lse, ref, lref)


@pytest.mark.parametrize("dk,dv", DIMS)
@pytest.mark.parametrize("nq", [50, 200])
@pytest.mark.parametrize("masked", [range(0, 4), range(4, 8), (0, 4), (0, 1, 2, 4, 6)])
def test_split_ranges(oracle, nq, dk, dv, masked):
    """Two key ranges of four blocks: one of them empty, or both without their first blocks."""
    x, q, k, v, ref = masked_inputs((1, 2, nq, 1024, dk, dv), "bf16", 128, masked)
    o = pkg.attn_fwd_splitkv(q, k, v, 2, x.scale)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    assert_close(o.float().cpu().numpy(), oracle.attn(*ref, x.scale), "bf16", f"{nq} {dk},{dv} {masked}")


def test_split_by_the_library_past_one_cta_per_sm(oracle):
    """80 heads in 3 ranges of d = 64: two one-tile CTAs an SM.  The first range has no key."""
    x, q, k, v, ref = masked_inputs((2, 40, 3, 9000, 64, 64), "bf16", 128, range(0, 24))
    o = pkg.attn_fwd_splitkv(q, k, v, pkg.MOA_SPLITS_AUTO, x.scale)
    assert_close(o.float().cpu().numpy(), oracle.attn(*ref, x.scale), "bf16", "80 heads")


@pytest.mark.parametrize("scale", [1.5, -0.2, -1.5])
@pytest.mark.parametrize("dtype,dk,dv", [("bf16", 64, 64), ("bf16", 128, 128), ("fp32", 64, 64)])
def test_other_scales(oracle, dtype, dk, dv, scale):
    """Scales of either sign, above and below 1: the masks are -inf times their sign."""
    value = -float("inf") if scale > 0 else float("inf")
    x, q, k, v, ref = masked_inputs((1, 2, 300, 500, dk, dv), dtype, 128, (0, 2), value)
    o, lse = pkg.attn_fwd_lse(q, k, v, scale)
    oref, lref = oracle.attn_lse(*ref, scale)
    assert_close(o.float().cpu().numpy(), oref, dtype, f"{scale}")
    check_lse(scale, lse, ref, lref)


@pytest.mark.parametrize("dtype,nk", [("fp32", 60), ("fp32", 300), ("bf16", 60), ("bf16", 300)])
@pytest.mark.parametrize("nq", [9, 600])
def test_no_key_at_all(nq, dtype, nk):
    x, q, k, v, _ = masked_inputs((1, 2, nq, nk, 64, 64), dtype, nk, (0,))
    o, lse = pkg.attn_fwd_lse(q, k, v, x.scale)
    assert torch.all(torch.isnan(o)) and torch.all(lse == float("-inf"))
