"""A (b, h) slice of a split call with a given number of ranges has the same bits alone and in a call
of any number of slices."""
import pytest

from gpu_helpers import to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402
from paper_2606_07713_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (128, 64), (64, 128)])
@pytest.mark.parametrize("nq", [7, 128, 130])
def test_slice_bits_with_a_given_number_of_ranges(nq, dk, dv):
    """80 slices in 5 ranges (more CTAs than two per SM) against 1 and 6 of them."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = I.make_inputs(I.custom_config(2, 40, nq, 1300, dk, dv, dtype="bf16", seed=nq + dk + dv))
    q, k, v = to_device(x)
    whole = pkg.attn_fwd_splitkv(q, k, v, 5, x.scale)
    for b, h, n in ((0, 0, 1), (1, 39, 1), (1, 10, 6)):
        one = [t[b:b + 1, h:h + n].contiguous() for t in (q, k, v)]
        assert torch.equal(pkg.attn_fwd_splitkv(*one, 5, x.scale), whole[b:b + 1, h:h + n])
