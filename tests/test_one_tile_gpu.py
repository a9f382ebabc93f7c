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
