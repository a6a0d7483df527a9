"""The state buffer is the whole state of a run in fp32 precision: what a caller writes into it between steps is what the
next step works from, and so is a projection that is set between two replays of a captured step."""
import pytest
import torch

from paper_2410_01623_b200 import binding as fb

pytestmark = pytest.mark.gpu

SHORT = [(200, 333), (333, 200)]
LONG = [(512, 1376), (1376, 512), (333, 901)] * 4           # above 5 Mi elements
CASES = [(SHORT, 64, torch.float32), (SHORT, 150, torch.float32), (LONG, 128, torch.float32), (LONG, 128, torch.bfloat16)]


def _run(shapes, r, dtype, seed, force):
    f = fb.Fira(shapes, r, dtype, fb.make_hparams(flags=fb.FLAG_FORCE_SIMT if force else 0))
    g = torch.Generator(device="cuda").manual_seed(seed)
    for i, (m, n) in enumerate(shapes):
        f.set_projection(i, torch.linalg.qr(torch.randn(min(m, n), r, generator=g, device="cuda"))[0].to(dtype).contiguous())
    W = [(torch.randn(m, n, generator=g, device="cuda") * 0.02).to(dtype) for m, n in shapes]
    G = [torch.randn(m, n, generator=g, device="cuda").to(dtype) for m, n in shapes]
    return f, W, G


def _scalars(shapes, r, dtype):
    """Offsets of the matrices' scalars: P, M, V and 32 bytes of scalars per matrix, each on a 256-byte boundary."""
    pad = lambda b: (b + 255) // 256 * 256                                              # noqa: E731
    es, at, out = 2 if dtype == torch.bfloat16 else 4, 0, []
    for m, n in shapes:
        at += pad(min(m, n) * r * es) + 2 * pad(max(m, n) * r * 4)
        out.append(at)
        at += 256
    return out


@pytest.mark.parametrize("shapes,r,dtype", CASES)
def test_a_checkpoint_copied_into_the_state_buffer_goes_on_from_there(shapes, r, dtype):
    force = len(shapes) > 2
    a, Wa, Ga = _run(shapes, r, dtype, 1, force)
    b, Wb, Gb = _run(shapes, r, dtype, 2, force)
    a.step(Wa, Ga)
    for _ in range(3):
        b.step(Wb, Gb)
    a.state.copy_(b.state)
    for at in _scalars(shapes, r, dtype):       # of the scalars the remembered norm (first) and the step count (last) are state
        a.state[at + 4:at + 24] = 0x7f
    for x, y in zip(Wa, Wb):
        x.copy_(y)
    for _ in range(2):
        a.step(Wa, Gb)
        b.step(Wb, Gb)
    for i in range(len(shapes)):
        assert torch.equal(Wa[i], Wb[i])
        for x, y in zip(a.get_state(i)[:2], b.get_state(i)[:2]):
            assert torch.equal(x, y)
        assert a.get_state(i)[2:] == b.get_state(i)[2:]


@pytest.mark.parametrize("shapes,r,dtype", CASES)
def test_replays_of_a_captured_step_use_the_projection_of_the_time(shapes, r, dtype):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        f, W, G = _run(shapes, r, dtype, 3, len(shapes) > 2)
        f.step(W, G)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            f.step(W, G)
        g = torch.Generator(device="cuda").manual_seed(4)
        for i, (m, n) in enumerate(shapes):
            f.set_projection(i, torch.linalg.qr(torch.randn(min(m, n), r, generator=g, device="cuda"))[0].to(dtype).contiguous())
        state, W0 = f.state.clone(), [w.clone() for w in W]
        graph.replay()
        replayed, after = [w.clone() for w in W], f.state.clone()
        f.state.copy_(state)
        for w, w0 in zip(W, W0):
            w.copy_(w0)
        f.step(W, G)
        stream.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(W, replayed))
        assert torch.equal(f.state, after)
        del graph
