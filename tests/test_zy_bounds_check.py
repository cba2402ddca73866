"""The debug build with range checks (RES2TAC_CHECK_BOUNDS): every checked global access of the
aggregation and WTA kernels stays inside its buffer on tiny and ragged shapes, every tuning and
both sum widths, and the maps still equal the oracle's. A failing check records its site and
skips the access (no trap), so a failure here shows as a nonzero site."""
import itertools

import numpy as np
import pytest

import oracle
from paper_2106_07927_gb300 import binding, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def check_lib():
    yield binding.use_check_library(True)
    binding.use_check_library(False)


def test_range_checks_pass_on_tiny_shapes(check_lib):
    import torch
    rng = np.random.default_rng(77)
    cases = [(1, 1, 16), (5, 3, 16), (17, 9, 32), (33, 20, 48), (70, 13, 64), (9, 40, 128),
             (130, 7, 144), (40, 31, 256)]
    # one plane per two directions and one per direction, 16-bit and 32-bit sums
    methods = ((120, 8), (16384, 8), (90, 4), (200, 8), (255, 4), (880, 8))
    for (W, H, D), (p2, paths) in itertools.product(cases, methods):
        left = rng.integers(0, 256, (H, W)).astype(np.uint8)
        right = rng.integers(0, 256, (H, W)).astype(np.uint8)
        prm = scenes.params(W, H, D, 9, 7, 10, p2, paths, 3)
        st = binding.Stereo(prm)
        assert binding.res2tac_bounds_status(st.handle)[0] == 1  # the debug build
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        ref = oracle.sgm(left, right, D, 9, 7, 10, p2, paths, 3)
        for sdpl, mode, cpl in itertools.product((8, 16, 32), (1, 2), (1, 2)):
            if D % sdpl:
                continue
            binding.res2tac_set_tuning(st.handle, binding.res2tac_tuning(0, 0, 0, sdpl, mode, cpl))
            out = st.compute(L, R)
            torch.cuda.synchronize()
            checked, site, off = binding.res2tac_bounds_status(st.handle)
            assert site == 0, (W, H, D, sdpl, mode, cpl, site, off)
            assert np.array_equal(binding.u16(out), ref), (W, H, D, sdpl, mode, cpl)
        if p2 <= 255:  # the selection's sub-pixel map
            binding.res2tac_set_tuning(st.handle, binding.res2tac_tuning())
            st.compute_subpixel(L, R)
            torch.cuda.synchronize()
            assert binding.res2tac_bounds_status(st.handle)[1] == 0, (W, H, D, p2, "subpixel")
        st.close()


@pytest.mark.parametrize("p2,paths", [(120, 8), (200, 8), (200, 4), (880, 8), (16384, 8)])
def test_range_checks_pass_in_batches(check_lib, p2, paths):
    import torch
    rng = np.random.default_rng(78)
    shapes = [(1, 1, 16), (5, 3, 16), (33, 20, 48), (31, 24, 48), (9, 40, 128), (130, 7, 144),
              (40, 31, 256), (300, 12, 64)] + [(40, 9, 32)] * 35
    prm = scenes.params(64, 64, 64, 9, 7, 10, p2, paths, 3)
    st = binding.Stereo(prm)
    keep, pairs, refs = [], [], []
    for W, H, D in shapes:
        left = rng.integers(0, 256, (H, W)).astype(np.uint8)
        right = rng.integers(0, 256, (H, W)).astype(np.uint8)
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        o = torch.full((H, W), -1, dtype=torch.int16, device="cuda")
        keep.append((L, R, o))
        pairs.append(binding.res2tac_pair(L.data_ptr(), R.data_ptr(), W, o.data_ptr(), 2 * W, W, H,
                                          D, 0))
        refs.append(oracle.sgm(left, right, D, 9, 7, 10, p2, paths, 3))
    binding.res2tac_compute_batch(st.handle, pairs, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    checked, site, off = binding.res2tac_bounds_status(st.handle)
    assert (checked, site) == (1, 0), (site, off)
    for (_, _, o), ref in zip(keep, refs):
        assert np.array_equal(binding.u16(o), ref)
    st.close()
