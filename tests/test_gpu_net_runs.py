"""The proposal net's kernels at the edges of their work split, against the FP64 oracle on
the GPU's own bf16 inputs (bounds of tests/test_gpu_net.py): one pixel, one row, images one
pixel short of, equal to and past a 128-pixel tile, and runs of a block that end within a
column of tiles and go on in the next column or frame (more tiles than resident blocks).
Parameter gradients into buffers that are only 4-byte aligned equal those into aligned ones
up to the order of FP32 additions."""
import numpy as np
import pytest

from oracle import net as onet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (2, 1, 300), (3, 2, 127), (1, 5, 128), (2, 7, 129), (1, 3, 258),
                                   (40, 33, 130)])
def test_layers_at_tile_edges(n, h, w):
    import torch
    from paper_2603_21055_gb300 import binding as B
    from paper_2603_21055_gb300.proposal import ProposalNet
    rng = np.random.default_rng(100 * h + w)
    params = [(x, rng.normal(0, 0.05, size=b.shape).astype(np.float32)) for x, b in onet.init_params(5)]
    net = ProposalNet(params)
    dev = lambda a: torch.as_tensor(a.astype(np.float32)).cuda()
    net.forward(dev(rng.uniform(size=(n, 3, h, w))), dev(rng.uniform(0.5, 4.0, size=(n, h, w))))
    net.loss_grad(dev(rng.normal(0, 0.01, size=(n, h, w))), dev(rng.normal(1, 0.5, size=(n, h, w))), logit_weight=0.5)
    net.backward()
    assert net.check() == 0
    bufs, px = net.buffers(), n * h * w

    def planar(ptr, c):
        a = net.workspace_array(ptr, px * c).float().cpu().numpy().astype(np.float64)
        return a.reshape(n, h, c // 8, w, 8).transpose(0, 1, 3, 2, 4).reshape(n, h, w, c)

    x = [planar(bufs.x[0], 16)] + [planar(bufs.x[l], 32) for l in (1, 2, 3)]
    y = net.workspace_array(bufs.y4, px * 2, torch.float32).cpu().numpy().astype(np.float64).reshape(n, h, w, 2)
    dy = [planar(bufs.dpre[l], 32) for l in range(3)] + [planar(bufs.dy4, 16)[..., :2]]
    near = lambda got, ref, mag, rel: np.all(np.abs(got - ref) <= rel * np.abs(ref) + 1e-5 * mag + 1e-30)
    mags = []
    for l in range(4):
        cin, cout = onet.CHANNELS[l], onet.CHANNELS[l + 1]
        xin, wq, b = x[l][..., :cin], onet.bf16(params[l][0]), params[l][1].astype(np.float64)
        ref = onet.conv3x3(xin, wq, b)
        mag = onet.conv3x3(np.abs(xin), np.abs(wq), np.abs(b))
        if l < 3:
            assert near(x[l + 1], np.maximum(ref, 0.0), mag, 2.0 ** -8), l
        else:
            assert near(y, ref, mag, 0.0)
        dx, dw, db = onet.conv3x3_backward(xin, wq, dy[l])
        dxa, dwa, dba = onet.conv3x3_backward(np.abs(xin), np.abs(wq), np.abs(dy[l]))
        if l > 0:
            assert near(dy[l - 1], dx * (xin > 0), dxa, 2.0 ** -8), l
        got = net.dw[l].cpu().numpy().astype(np.float64)[:, :cin, :cout].reshape(3, 3, cin, cout)
        assert np.all(np.abs(got - dw) <= 1e-4 * dwa + 1e-30), l
        assert np.all(np.abs(net.db[l].cpu().numpy()[:cout] - db) <= 1e-4 * dba + 1e-30), l
        mags.append((dwa, dba))
    # the same into buffers one float past an aligned address
    odd_w, odd_b = ([torch.full((t.numel() + 1,), float("nan"), device="cuda") for t in ts] for ts in (net.dw, net.db))
    g = B.sgad_net_grads()
    for l in range(4):
        g.dw[l], g.db[l] = odd_w[l].data_ptr() + 4, odd_b[l].data_ptr() + 4
    B.sgad_net_backward(net._params, g, n, h, w, net.workspace.data_ptr(), net.workspace.numel(), net.stream())
    assert net.check() == 0
    for l in range(4):
        cin, cout = onet.CHANNELS[l], onet.CHANNELS[l + 1]
        d = (odd_w[l][1:].view_as(net.dw[l]) - net.dw[l]).double().abs().cpu().numpy()
        assert np.all(d[:, :cin, :cout].reshape(3, 3, cin, cout) <= 2e-4 * mags[l][0] + 1e-30), l
        assert np.all((odd_b[l][1:] - net.db[l]).double().abs().cpu().numpy()[:cout] <= 2e-4 * mags[l][1] + 1e-30), l
