"""Path planes (P2 <= 255): every lane count of the sheared chains, one plane per pair of opposite
directions (2 P2 <= 255) and one per direction, against the oracle, bit by bit; and the batch route
on them at its limits of group size and scratch."""
import numpy as np
import pytest

import oracle
from paper_2106_07927_gb300 import binding, scenes

pytestmark = pytest.mark.gpu


def _pair(seed, W, H, D):
    left, right, _ = scenes.make_scene(("road", "nadir")[seed % 2], seed, W, H, D)
    return left, right


# D / 16 = 1 .. 16 lanes per chain, with the row path's 2, 4 and 8 disparities per lane; images
# narrower than D, than a warp's chains and than two row chunks; P2 at the byte limits 127, 128, 255.
@pytest.mark.parametrize("D", range(16, 257, 16))
@pytest.mark.parametrize("W,H,p2,paths", [(61, 23, 127, 8), (40, 9, 128, 8), (9, 40, 255, 4),
                                          (131, 6, 127, 4), (1, 5, 255, 8)])
def test_planes_match_oracle(D, W, H, p2, paths):
    import torch
    rng = np.random.default_rng(D + W)
    left = rng.integers(0, 256, (H, W)).astype(np.uint8)
    right = np.roll(left, -3, axis=1)
    prm = scenes.params(W, H, D, 9, 7, 11, p2, paths, 3)
    ref, dbg = oracle.sgm(left, right, D, 9, 7, 11, p2, paths, 3, 1, debug=True)
    st = binding.Stereo(prm)
    L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
    for dpl, sdpl in ((2, 16), (4, 8), (8, 16), (8, 8)):  # 8: one sheared chain per warp
        if D // dpl > 32:
            continue
        binding.res2tac_set_tuning(st.handle, binding.res2tac_tuning(agg_dpl=dpl, shear_dpl=sdpl))
        out = st.compute(L, R)
        got = st.debug_outputs()
        torch.cuda.synchronize()
        assert np.array_equal(got["cost"].cpu().numpy(), dbg["cost"])
        for k in ("agg", "dl", "dr"):
            assert np.array_equal(binding.u16(got[k]), dbg[k]), (k, dpl)
        assert np.array_equal(binding.u16(out), ref), dpl
    st.close()


@pytest.mark.parametrize("p2", [120, 200])
def test_batch_groups_and_scratch_limits(p2):
    import torch
    # 40 pairs of one size (more than a group holds), two of another D, one large one
    shapes = [(50, 30, 32)] * 40 + [(70, 20, 48)] * 2 + [(300, 200, 128)]
    prm = scenes.params(64, 64, 64, 9, 7, 10, p2, 8, 3)
    pairs, outs, want, keep = [], [], [], []
    for i, (W, H, D) in enumerate(shapes):
        left, right = _pair(i, W, H, D)
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        o = torch.full((H, W), -1, dtype=torch.int16, device="cuda")
        keep.append((L, R))
        outs.append(o)
        pairs.append(binding.res2tac_pair(L.data_ptr(), R.data_ptr(), W, o.data_ptr(), 2 * W, W, H,
                                          D, 0))
        want.append(oracle.sgm(left, right, D, 9, 7, 10, p2, 8, 3))
    params = binding.params_from_dict(prm)
    one = binding.res2tac_batch_workspace_bytes(params, pairs[-1:])
    # grown on demand; reserved for the batch; reserved for the large pair alone
    for reserve, batch in ((0, pairs), (binding.res2tac_batch_workspace_bytes(params, pairs), pairs),
                           (one, pairs[-1:])):
        ctx = binding.Stereo(prm)
        if reserve:
            binding.res2tac_batch_reserve(ctx.handle, reserve, len(batch))
        for o in outs:
            o.fill_(-1)
        # twice, on two streams: the second call uses the same scratch
        s2 = torch.cuda.Stream()
        s2.wait_stream(torch.cuda.current_stream())
        binding.res2tac_compute_batch(ctx.handle, batch, torch.cuda.current_stream().cuda_stream)
        binding.res2tac_compute_batch(ctx.handle, batch, s2.cuda_stream)
        torch.cuda.synchronize()
        for o, w in list(zip(outs, want))[-len(batch):]:
            assert np.array_equal(binding.u16(o), w)
        ctx.close()


# pairs that a scratch of the size callers reserve holds at once: one launch per stage and group
@pytest.mark.parametrize("n,W,H,D,p2,paths,groups", [
    (5, 160, 120, 32, 200, 8, 1), (3, 160, 120, 32, 100, 8, 1), (2, 160, 120, 32, 100, 4, 1),
    (8, 320, 240, 128, 200, 8, 4), (5, 640, 480, 64, 100, 8, 5), (33, 40, 24, 16, 120, 8, 2)])
def test_reserved_small_batches_run_at_once(n, W, H, D, p2, paths, groups):
    import torch
    prm = scenes.params(64, 64, 64, 9, 7, 10, p2, paths, 3)
    keep, pairs, outs = [], [], []
    for i in range(n):
        L, R = (torch.from_numpy(a).cuda() for a in _pair(i % 4, W, H, D))
        o = torch.full((H, W), -1, dtype=torch.int16, device="cuda")
        keep.append((L, R))
        outs.append(o)
        pairs.append(binding.res2tac_pair(L.data_ptr(), R.data_ptr(), W, o.data_ptr(), 2 * W, W, H,
                                          D, 0))
    ctx = binding.Stereo(prm)
    binding.res2tac_batch_reserve(ctx.handle, binding.res2tac_batch_workspace_bytes(
        binding.params_from_dict(prm), pairs), n)
    binding.res2tac_compute_batch(ctx.handle, pairs, torch.cuda.current_stream().cuda_stream)
    assert binding.res2tac_last_launch_count(ctx.handle) == 6 * groups
    single = binding.Stereo(scenes.params(W, H, D, 9, 7, 10, p2, paths, 3))
    want = [single.compute(*k) for k in keep]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, outs))
    single.close()
    ctx.close()


def test_settings_off_the_planes_take_the_values_of_the_sums():
    import torch
    W, H, D = 200, 110, 128
    left, right = _pair(3, W, H, D)
    ref = oracle.sgm(left, right, D, 9, 7, 10, 120, 8, 3)
    L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
    st = binding.Stereo(scenes.params(W, H, D, 9, 7, 10, 120, 8, 3))
    # (shear_dpl, shear_cpl) that a partly given setting ends up with
    for given, want in ((dict(wta_chunk=64), (8, 1)), (dict(cost_mode=2), (16, 2)),
                        (dict(row_mode=1), (16, 2)), (dict(row_cost=2), (16, 2)),
                        (dict(shear_cpl=2), (16, 2)), (dict(shear_dpl=32), (32, 2)),
                        (dict(cost_mode=2, shear_cpl=1), (16, 1)), (dict(), (8, 1))):
        binding.res2tac_set_tuning(st.handle, binding.res2tac_tuning(**given))
        t = binding.res2tac_get_tuning(st.handle)
        assert (t.shear_dpl, t.shear_cpl) == want, given
        out = st.compute(L, R)
        torch.cuda.synchronize()
        assert np.array_equal(binding.u16(out), ref), given
    st.close()


def test_reported_sizes_cover_what_contexts_hold():
    import torch
    W, H, D = 500, 300, 128
    left, right = _pair(2, W, H, D)
    L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
    out = torch.empty((H, W), dtype=torch.int16, device="cuda")
    binding.Stereo(scenes.params(16, 16, 16, 9, 7, 10, 120, 8, 3)).close()  # the library is loaded
    # planes (two methods), exact check, 32-bit sums, NCC
    for p2, flags, n, planes in ((120, 3, 9, 4), (200, 7, 9, 8), (16384, 3, 9, 0),
                                 (880, 3 | 8, 5, 0)):
        prm = scenes.params(W, H, D, n, 7 if n == 9 else 5, 10, p2, 8, flags)
        p = binding.params_from_dict(prm)
        need = binding.res2tac_workspace_bytes(p)
        torch.cuda.synchronize()
        maps = []
        for compact in (True, False):
            free = torch.cuda.mem_get_info()[0]
            st = binding.Stereo(prm, compact=compact)
            held = binding.res2tac_context_bytes(st.handle)
            took = free - torch.cuda.mem_get_info()[0]
            assert abs(took - held) <= 16 << 20  # the allocator's granularity
            if compact or not planes:
                assert 0.9 * need < held <= need
            else:
                assert held >= (1 + planes) * W * H * D > need
            maps.append(st.compute(L, R))
            if compact and p2 <= 255 and not flags & 4:
                pairs = [binding.res2tac_pair(L.data_ptr(), R.data_ptr(), W, out.data_ptr(), 2 * W,
                                              W, H, D, 0)]
                batch = binding.res2tac_batch_workspace_bytes(p, pairs)
                for reserve in (False, True):
                    if reserve:
                        binding.res2tac_batch_reserve(st.handle, batch, 1)
                    out.fill_(-1)
                    binding.res2tac_compute_batch(st.handle, pairs,
                                                  torch.cuda.current_stream().cuda_stream)
                    torch.cuda.synchronize()
                    assert torch.equal(out, maps[0])
                    assert binding.res2tac_context_bytes(st.handle) - held <= batch + 4096
            torch.cuda.synchronize()
            st.close()
        assert torch.equal(maps[0], maps[1])
        assert np.array_equal(binding.u16(maps[0]), oracle.sgm(
            left, right, D, prm["census_w"], prm["census_h"], 10, p2, 8, flags))
