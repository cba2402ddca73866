"""Calls captured into a CUDA graph: a replay on other images gives the maps of plain calls, and
later batches leave the scratch a captured batch uses where it is."""
import numpy as np
import pytest

import oracle
from paper_2106_07927_gb300 import binding, scenes

pytestmark = pytest.mark.gpu


def _pair(seed, W, H, D):
    left, right, _ = scenes.make_scene(("road", "nadir")[seed % 2], seed, W, H, D)
    return left, right


def _captured(torch, call):
    """Runs call once (warm-up), then captures it; returns the graph."""
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


# one chain per warp and 16 disparities per lane, one plane per two directions and per direction, the
# exact check (two passes), sums in place (32-bit ones) and the NCC cost
@pytest.mark.parametrize("W,H,D,p2,flags,cw,ch", [
    (160, 96, 64, 120, 3, 9, 7), (420, 40, 128, 200, 3, 9, 7), (160, 96, 64, 120, 7, 9, 7),
    (160, 96, 64, 16384, 3, 9, 7), (160, 96, 64, 880, 3 | 8, 5, 5)])
def test_captured_call_replays(W, H, D, p2, flags, cw, ch):
    import torch
    st = binding.Stereo(scenes.params(W, H, D, cw, ch, 10, p2, 8, flags))
    L, R = (torch.from_numpy(a).cuda() for a in _pair(1, W, H, D))
    out = torch.empty((H, W), dtype=torch.int16, device="cuda")
    g = _captured(torch, lambda: st.compute(L, R, out))
    for seed in (2, 3):
        left, right = _pair(seed, W, H, D)
        L.copy_(torch.from_numpy(left))
        R.copy_(torch.from_numpy(right))
        out.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(binding.u16(out),
                              oracle.sgm(left, right, D, cw, ch, 10, p2, 8, flags))
    del g
    st.close()


@pytest.mark.parametrize("p2", [120, 200])
def test_captured_batch_keeps_its_scratch(p2):
    import torch
    shapes = [(300, 100, 64)] * 10 + [(96, 60, 128), (200, 50, 256)]
    ctx = binding.Stereo(scenes.params(64, 64, 64, 9, 7, 10, p2, 8, 3))
    images = [[torch.from_numpy(a).cuda() for a in _pair(i, *s)] for i, s in enumerate(shapes)]
    outs = [torch.empty((H, W), dtype=torch.int16, device="cuda") for W, H, D in shapes]

    def descriptors(ims, maps, sizes):
        return [binding.res2tac_pair(a.data_ptr(), b.data_ptr(), W, o.data_ptr(), 2 * W, W, H, D, 0)
                for (a, b), o, (W, H, D) in zip(ims, maps, sizes)]

    pairs = descriptors(images, outs, shapes)
    batch = lambda ps: binding.res2tac_compute_batch(ctx.handle, ps,
                                                     torch.cuda.current_stream().cuda_stream)
    # an earlier batch sized the scratch
    tall = [(300, 100, 64)] * 12 + [(300, 200, 64)] * 3
    ims = [[torch.from_numpy(a).cuda() for a in _pair(40 + i, *s)] for i, s in enumerate(tall)]
    maps = [torch.empty((H, W), dtype=torch.int16, device="cuda") for W, H, D in tall]
    batch(descriptors(ims, maps, tall))
    g = _captured(torch, lambda: batch(pairs))
    # a lone pair whose sums fit what that batch needs and whose planes (5 or 9 bytes per estimate) do
    # not
    prm = binding.params_from_dict(scenes.params(64, 64, 64, 9, 7, 10, p2, 8, 3))
    held = binding.res2tac_batch_workspace_bytes(prm, descriptors(ims, maps, tall))
    W, D = 640, 128
    H = next(h for h in range(1, 2000) if h * W * (5 * D + 25) > 1.02 * held)
    assert H * W * (3 * D + 25) < 0.8 * held
    lone = [torch.from_numpy(a).cuda() for a in _pair(77, W, H, D)]
    lone_out = torch.empty((H, W), dtype=torch.int16, device="cuda")
    before = binding.res2tac_context_bytes(ctx.handle)
    batch(descriptors([lone], [lone_out], [(W, H, D)]))
    torch.cuda.synchronize()
    # the scratch stayed where the graph has it
    assert binding.res2tac_context_bytes(ctx.handle) == before
    for i, s in enumerate(shapes):
        left, right = _pair(100 + i, *s)
        images[i][0].copy_(torch.from_numpy(left))
        images[i][1].copy_(torch.from_numpy(right))
        outs[i].fill_(-1)
    g.replay()
    torch.cuda.synchronize()
    for i, (w, h, d) in enumerate(shapes):
        left, right = _pair(100 + i, w, h, d)
        assert np.array_equal(binding.u16(outs[i]), oracle.sgm(left, right, d, 9, 7, 10, p2, 8, 3))
    single = binding.Stereo(scenes.params(W, H, D, 9, 7, 10, p2, 8, 3))
    want = single.compute(*lone)
    torch.cuda.synchronize()
    assert torch.equal(want, lone_out)
    # a call under capture allocates nothing either
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2):
        batch(descriptors([lone], [lone_out], [(W, H, D)]))
    lone_out.fill_(-1)
    g2.replay()
    torch.cuda.synchronize()
    assert torch.equal(want, lone_out)
    del g, g2
    single.close()
    ctx.close()
