"""Every kernel route under stream capture (twice in one graph, replayed) and interleaved over three
streams: the bits of the call made alone.  The kernels of a call, and of calls that follow one another,
are launched as dependent ones; the backward calls of one stream share a workspace here, so that a
kernel that starts before the one before it has ended would show."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_2606_07713_gb300 as pkg  # noqa: E402

BF, F32 = torch.bfloat16, torch.float32


def rnd(gen, *shape, dtype=BF):
    return torch.randn(shape, device="cuda", generator=gen).to(dtype)


def routes():
    """name -> call(workspace) -> outputs."""
    gen = torch.Generator(device="cuda").manual_seed(1)
    cases = {}
    for B, H, N, M, d, dv, t in [
            (1, 2, 128, 128, 64, 64, F32), (2, 4, 300, 500, 64, 64, F32), (16, 12, 197, 197, 64, 64, BF),
            (2, 4, 700, 900, 128, 128, BF), (10, 16, 385, 300, 128, 64, BF), (10, 16, 385, 300, 64, 64, BF),
            (2, 3, 50, 3000, 64, 64, BF), (8, 4, 1, 4097, 128, 128, BF)]:
        q, k, v = (rnd(gen, B, H, n, w, dtype=t) for n, w in ((N, d), (M, d), (M, dv)))
        g = rnd(gen, B, H, N, dv, dtype=t)
        o, lse = pkg.attn_fwd_lse(q, k, v)
        name = f"{B}x{H}x{N}x{M} {d},{dv} {t}"
        cases["fwd " + name] = lambda ws, a=(q, k, v): tuple(pkg.attn_fwd_lse(*a))
        if t is BF:
            cases["split " + name] = lambda ws, a=(q, k, v): (pkg.attn_fwd_splitkv(*a), pkg.attn_fwd_splitkv(*a, 5))
        cases["bwd " + name] = lambda ws, a=(q, k, v, o, lse, g): tuple(pkg.attn_bwd(*a, workspace=ws))
        if t is BF and d == dv == 64:
            # dQ's last bits vary from run to run
            cases["fused " + name] = lambda ws, a=(q, k, v, o, lse, g): tuple(
                pkg.attn_bwd(*a, workspace=ws, fused=True))[1:]
    for N in (1, 300):
        x, w = rnd(gen, 2, N, 512), rnd(gen, 512, 3 * 8 * 64) / 23
        cases[f"qkv {N}"] = lambda ws, a=(x, w): tuple(pkg.qkv_proj(*a, 8, 64, 64))
    return cases


@pytest.fixture(scope="module")
def cases():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    calls = routes()
    torch.cuda.synchronize()
    want = {}
    for name, call in calls.items():
        want[name] = call(workspace())
        torch.cuda.synchronize()
    return calls, want


def workspace():
    return torch.empty(64 << 20, dtype=torch.uint8, device="cuda")


def test_capture_and_replay(cases):
    calls, want = cases
    ws = workspace()
    for name, call in calls.items():
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            got = call(ws) + call(ws)
        for _ in range(3):
            for t in got:
                t.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, want[name] + want[name])), name
    pkg.check(pkg.get_device_status())


def test_interleaved_streams(cases):
    calls, want = cases
    streams = [(torch.cuda.Stream(), workspace()) for _ in range(3)]
    torch.cuda.synchronize()
    got = []
    for turn in range(4):
        for i, (name, call) in enumerate(calls.items()):
            stream, ws = streams[(i + turn) % 3]
            with torch.cuda.stream(stream):
                got.append((name, call(ws)))
    torch.cuda.synchronize()
    for name, out in got:
        assert all(torch.equal(a, b) for a, b in zip(out, want[name])), name
    pkg.check(pkg.get_device_status())
