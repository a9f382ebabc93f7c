"""The projection's tiles at their edges.  Inputs are small integers, so every product and sum is
exact in fp32 whatever the order, and the outputs must be the exact sums rounded once to bf16."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.lib()


SHAPES = [  # B, N, d_model, H, d_k, d_v
    (1, 1, 8, 1, 64, 64),         # one token, one feature step, 192 columns
    (3, 5, 4096, 2, 64, 64),      # 15 tokens, the widest split of d
    (1, 16, 72, 3, 64, 64),       # a full 16-token tile, a feature tail
    (1, 17, 520, 1, 128, 64),     # one token past it
    (2, 32, 328, 5, 64, 128),     # 64 tokens
    (5, 13, 1000, 7, 128, 128),   # 65 tokens
    (1, 128, 2048, 4, 64, 64),    # the last size of the small tile
    (3, 43, 192, 1, 64, 64),      # 129 tokens: the first of the pair tile, columns in halves
    (1, 256, 64, 2, 128, 128),    # a full pair tile
    (1, 257, 136, 3, 128, 64),    # one token past it: the second CTA's rows are empty
    (2, 600, 1000, 20, 64, 64),   # sequences that end inside a tile, 75 tiles for the pairs
    (4, 2048, 256, 16, 64, 64),   # more than one round, the last one in halves
    (1, 9000, 128, 9, 128, 64),   # token blocks past a whole group
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_projection_tiles_exact(shape):
    B, N, d, H, dk, dv = shape
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    x = torch.randint(-3, 4, (B, N, d), generator=g, device="cuda").to(torch.bfloat16)
    w = torch.randint(-3, 4, (d, H * (2 * dk + dv)), generator=g, device="cuda").to(torch.bfloat16)
    out = pkg.qkv_proj(x, w, H, dk, dv)
    torch.cuda.synchronize()
    pkg.check(pkg.get_device_status())
    ref = (x.double().reshape(B * N, d) @ w.double()).float().to(torch.bfloat16)
    c0 = 0
    for name, t, dim in zip("QKV", out, (dk, dk, dv)):
        want = ref[:, c0:c0 + H * dim].reshape(B, N, H, dim).permute(0, 2, 1, 3)
        assert torch.equal(t, want), f"{shape} {name}"
        c0 += H * dim
