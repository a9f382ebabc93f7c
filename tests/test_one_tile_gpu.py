"""Calls of at most 128 query rows (one Q tile per CTA), whole and with a split key axis, and the
merge of more key ranges than a warp has lanes."""
import pytest

from gpu_helpers import assert_close, to_device

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
@pytest.mark.parametrize("nq", [1, 33, 127, 128])
def test_one_tile_matches_two_tiles_and_oracle(oracle, nq, dk, dv):
    """The first nq rows of a 200-row call (two tiles where d > 64) are the nq-row call's rows bit
    for bit: a row's arithmetic does not depend on its CTA's tiles.  The split calls (2 ranges, and
    one per key block) stay within the bf16 bound."""
    x = I.make_inputs(I.custom_config(2, 3, 200, 1029, dk, dv, dtype="bf16", seed=nq + dk + 2 * dv))
    q, k, v = to_device(x)
    qs = q[:, :, :nq].contiguous()
    o = pkg.attn_fwd(qs, k, v, x.scale)
    assert torch.equal(o, pkg.attn_fwd(q, k, v, x.scale)[:, :, :nq])
    ref = oracle.attn(x.q[:, :, :nq], x.k, x.v, x.scale)
    for splits in (1, 2, 9):
        o = pkg.attn_fwd_splitkv(qs, k, v, splits, x.scale)
        torch.cuda.synchronize()
        pkg.check(pkg.get_device_status())
        assert_close(o.float().cpu().numpy(), ref, "bf16", f"nq={nq} {dk},{dv} splits={splits}")


@pytest.mark.parametrize("nq,dv", [(5, 64), (130, 128)])
def test_merge_of_many_ranges(oracle, nq, dv):
    """33 and 65 key ranges: one and two ranges past the lanes of the merge's warp."""
    x = I.make_inputs(I.custom_config(1, 2, nq, 65 * 128, 128, dv, dtype="bf16", seed=nq + dv))
    q, k, v = to_device(x)
    ref = oracle.attn(x.q, x.k, x.v, x.scale)
    for splits in (33, 65):
        o = pkg.attn_fwd_splitkv(q, k, v, splits, x.scale)
        torch.cuda.synchronize()
        pkg.check(pkg.get_device_status())
        assert_close(o.float().cpu().numpy(), ref, "bf16", f"nq={nq} splits={splits}")


@pytest.mark.parametrize("bh", [2, 40])
@pytest.mark.parametrize("nk", [1029, 1280])
def test_d64_split_small_and_large_grids(oracle, bh, nk):
    """Two tiles on the same rows up to one CTA per SM, one-tile CTAs two to an SM past it (40 x 5
    ranges), with an odd and an even number of key blocks in the last range."""
    x = I.make_inputs(I.custom_config(1, bh, 7, nk, 64, 64, dtype="bf16", seed=bh + nk))
    q, k, v = to_device(x)
    o = pkg.attn_fwd_splitkv(q, k, v, 5, x.scale)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    assert_close(o.float().cpu().numpy(), oracle.attn(x.q, x.k, x.v, x.scale), "bf16", f"{bh}x{nk}")


@pytest.mark.parametrize("masked", [range(1, 8, 2), range(0, 8, 2), (1, 2, 3, 5), (0, 3, 4, 7)])
@pytest.mark.parametrize("dk", [64, 128])
def test_blocks_of_masked_keys(oracle, dk, masked):
    """Keys whose score is -inf (first feature: 1 in Q, -inf in K) have no part in the result, also
    where one of a CTA's two tiles has no other keys (every odd or even block of a range)."""
    x = I.make_inputs(I.custom_config(1, 2, 50, 1024, dk, 64, dtype="bf16", seed=dk))
    q, k, v = to_device(x)
    q[..., 0] = 1.0
    k[..., 0] = 0.0
    keep = [i for i in range(1024) if i // 128 not in masked]
    km = torch.full_like(k[..., 0], float("-inf"))
    km[..., keep] = 0.0
    k[..., 0] = km
    o = pkg.attn_fwd_splitkv(q, k, v, 2, x.scale)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    f = [t.float().cpu().numpy().astype("float64") for t in (q, k[:, :, keep], v[:, :, keep])]
    assert_close(o.float().cpu().numpy(), oracle.attn(*f, x.scale), "bf16", f"{dk} {masked}")
