"""The library's launches overlap the end of the kernel before them; the effects must be those
of one kernel after another. Calls issued back to back on one stream, with the caller's own
kernels changing their inputs in between, give bit for bit what the same calls give with a
synchronisation after each; on the current stream, on a side stream and replayed from a graph.
Renderings and the proposal net's outputs are compared (their kernels add in a fixed order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem():
    import torch
    from paper_2603_21055_gb300 import splat
    from paper_2603_21055_gb300.proposal import ProposalNet
    from paper_2603_21055_gb300.synth import Camera
    gen = torch.Generator(device="cuda").manual_seed(2)
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    cam = Camera(40, 30, 40.0, 40.0, 20.0, 15.0, eye)
    kf = splat.DeviceKeyframe(cam, 2.0 + rnd(30, 40), torch.zeros(30, 40, device="cuda"), rnd(3, 30, 40),
                              rnd(30, 40), 0.03 + 0.03 * rnd(30, 40), True)
    sp = splat.Splatter()
    sp.plan([kf], [cam], slack=2.0)
    return sp, kf, cam, splat.alloc_images([cam]), ProposalNet(), rnd(1, 3, 30, 40), rnd(1, 30, 40)


def _run(sync, stream, graph):
    import torch
    sp, kf, cam, im, net, rgb, depth = _problem()
    steps, out = 12, []
    n = torch.zeros(1, device="cuda")
    delta, logit = torch.empty(1, 30, 40, device="cuda"), torch.empty(1, 30, 40, device="cuda")

    def step():
        n.add_(1.0)
        kf.offset.copy_(0.02 * torch.sin(n + kf.depth))            # the caller's kernels write the inputs
        kf.rgb.mul_(0.97)
        sp.forward([kf], [cam], im)
        net.forward(torch.cat([im[0]["rgb"][None]]), depth, delta, logit)
        if sync:
            torch.cuda.synchronize()
        return [im[0]["rgb"].clone(), im[0]["depth"].clone(), im[0]["alpha"].clone(), delta.clone(), logit.clone()]

    s = torch.cuda.Stream() if stream or graph else torch.cuda.current_stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        if graph:
            keep = (n.clone(), kf.rgb.clone())
            step()                                                  # warm-up
            n.copy_(keep[0])
            kf.rgb.copy_(keep[1])
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                kept = step()
            for _ in range(steps):
                g.replay()
                out.append([t.clone() for t in kept])
        else:
            out = [step() for _ in range(steps)]
    torch.cuda.synchronize()
    assert sp.check()[0] == 0 and net.check() == 0
    return [[t.cpu() for t in o] for o in out]


@pytest.mark.parametrize("stream,graph", [(False, False), (True, False), (True, True)])
def test_back_to_back_calls_equal_synchronised_ones(stream, graph):
    import torch
    want, got = _run(True, False, False), _run(False, stream, graph)
    for a, b in zip(want, got):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
    assert not torch.equal(want[0][0], want[1][0])
