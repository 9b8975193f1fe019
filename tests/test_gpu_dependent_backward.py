"""Back-to-back calls against synchronised ones (see test_gpu_dependent_launches.py) for the
rest of the library's launches: both losses, the splatting backward with a pose gradient, Adam,
the net's loss and backward, and the tracking of a frame. Every step's inputs are written by the
caller's kernels just before it and its outputs kept. Image gradients, Adam's results and the
tracked poses are equal bit for bit (their sums have a fixed order); sums by atomics up to the
order of FP32 additions (1e-5 of their norm, as in tests/test_gpu_batching.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(sync):
    import torch
    from paper_2603_21055_gb300 import binding as B
    from paper_2603_21055_gb300 import splat
    from paper_2603_21055_gb300.gicp import GicpTracker
    from paper_2603_21055_gb300.proposal import ProposalNet
    from paper_2603_21055_gb300.synth import Camera
    gen = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    new = lambda *s: torch.empty(*s, device="cuda")
    h, w = 45, 60
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    cam = Camera(w, h, 60.0, 60.0, 30.0, 22.0, eye)
    u, v = torch.meshgrid(torch.arange(w, device="cuda"), torch.arange(h, device="cuda"), indexing="xy")
    depth0 = 2.0 + 0.3 * torch.sin(0.2 * u) * torch.cos(0.3 * v) + 0.002 * rnd(h, w)
    kf = splat.DeviceKeyframe(cam, depth0.clone(), torch.zeros(h, w, device="cuda"), rnd(3, h, w), rnd(h, w),
                              depth0 / 60.0, True)
    sp = splat.Splatter()
    sp.plan([kf], [cam], slack=2.0)
    im = splat.alloc_images([cam])
    trgb, d_rgb, d_dep, pose = [rnd(3, h, w)], [new(3, h, w)], [new(h, w)], new(12)
    loss, valid = torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    grads = [dict(d_offset=new(h, w), d_rgb=new(3, h, w), d_logit=new(h, w), d_scale=new(h, w))]
    param, m, vv = rnd(3, h, w), torch.zeros(3, h, w, device="cuda"), torch.zeros(3, h, w, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    adam = (B.sgad_adam_tensor * 1)(B.sgad_adam_tensor(param.data_ptr(), d_rgb[0].data_ptr(), m.data_ptr(),
                                                       vv.data_ptr(), param.numel(), 0.01, B.SGAD_ADAM_PLAIN))
    net, rgb_in, d_in, t_d, t_l = ProposalNet(), rnd(1, 3, h, w), new(1, h, w), 0.01 * rnd(1, h, w), rnd(1, h, w)
    tr = GicpTracker(src_capacity=4096, map_capacity=1 << 15, stride=1, k_cov=6, max_iters=4, tol=0.0)
    step = torch.zeros(1, device="cuda")
    depth = depth0.clone()
    tr.frame(cam, depth)
    tr.set_pose(eye)
    tr.insert()
    torch.cuda.synchronize()
    out = []
    done = torch.cuda.synchronize if sync else (lambda: None)
    for _ in range(10):
        step.add_(1.0)
        kf.offset.copy_(0.02 * torch.sin(step + depth0))
        kf.rgb.mul_(0.97)
        sp.forward([kf], [cam], im)
        done()
        loss.zero_()
        sp.l1_loss_grad([cam], im, trgb, [depth0], 0.8, 1.0, d_rgb, d_dep, loss, valid)
        done()
        sp.ssim_loss_grad([cam], im, trgb, 0.2, d_rgb, loss)
        done()
        sp.backward([kf], [cam], [dict(rgb=d_rgb[0], depth=d_dep[0], pose=pose)], grads)
        done()
        B.sgad_adam_step_multi(adam, 0.9, 0.999, 1e-8, count.data_ptr(), sp.stream())
        done()
        torch.add(depth0[None], 0.01 * step, out=d_in)
        net.forward(rgb_in, d_in)
        done()
        net.loss_grad(t_d, t_l)
        done()
        net.backward()
        done()
        depth.copy_(depth0 + 0.003 * step)
        tr.frame(cam, depth)
        done()
        tr.track(eye)
        done()
        exact = [d_rgb[0].clone(), d_dep[0].clone(), param.clone(), m.clone(), tr.ws[:144].clone()]
        near = [g.clone() for g in grads[0].values()] + [pose.clone(), loss.clone(), net.loss.clone()]
        near += [t.clone() for t in net.dw + net.db]
        tr.insert()
        done()
        out.append((exact + [tr.map.count.clone()], near))
    torch.cuda.synchronize()
    assert sp.check()[0] == 0 and net.check() == 0 and tr.result()[1].status == 0
    return [([t.cpu() for t in a], [t.double().cpu() for t in b]) for a, b in out]


def test_back_to_back_calls_equal_synchronised_ones():
    import torch
    want, got = _run(True), _run(False)
    for (we, wn), (ge, gn) in zip(want, got):
        for i, (x, y) in enumerate(zip(we, ge)):
            assert torch.equal(x, y), i
        for i, (x, y) in enumerate(zip(wn, gn)):
            assert (x - y).norm() <= 1e-5 * x.norm(), i
    assert not torch.equal(want[0][0][0], want[1][0][0])
