"""Host models of the walks on path planes (csrc/planar.cuh): every cost copy and every store of a
sheared chain, with its restarts, against the chain definition; the row walk's chunks; and the
scan ranges of the selection's diagonals against the definition of D^R. The constants, ring sizes,
tiles, lane offsets and the rule for the sheared chains' shape are the header's own, printed by
planar_host.cu."""
import itertools
import os
import subprocess

import pytest

from paper_2106_07927_gb300 import build

NEVER = 1 << 30


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    """{first word: {key numbers: last number(s)}} of what planar_host.cu prints."""
    exe = str(tmp_path_factory.mktemp("host") / "planar_host")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "planar_host.cu")
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-o", exe, src], check=True)
    keys = {"const": 0, "shear_smem": 0, "mid": 1, "ring": 2, "tile": 2, "words": 1, "at": 3,
            "lanes": 2, "shape": 3}
    out = {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n"):
        if line:
            word, *v = line.split()
            v = tuple(map(int, v))
            k = keys[word]
            out.setdefault(word, {})[v[:k]] = v[k:] if len(v) - k > 1 else v[k]
    return out


def _walk(W, H, kind, j, paired, GS, PF):
    """(copies, stores, restarts) of one chain alone in its warp, pixel by pixel, as the kernel's
    two pointers and its fast and general groups of GS steps make them, in one part or (directions
    that share a plane) in two; copies are listed by the step that uses them. GS: steps of a group,
    PF: steps between a cost copy and its use."""
    sh = 0 if kind < 2 else (1 if kind < 4 else -1)
    back = kind & 1
    dy, dx = (-1, -sh) if back else (1, sh)
    ystart = H - 1 if back else 0
    x = (j + sh * ystart) % W
    stride, wrap = dy * W + dx, dx * W
    wp = ystart * W + x
    tw = NEVER if dx == 0 else (W - x if dx > 0 else x + 1)
    copies, stores, restarts = [], [], []
    base = 0
    for ph in range(2 if paired else 1):
        n = H if not paired else (H // 2 if (ph == 0) != bool(back) else H - H // 2)
        rp, tr = wp, tw
        tail = 0 if n < PF + GS else (n - PF) & ~(GS - 1)

        def copy_step(t):
            nonlocal rp, tr
            if t < n:
                if tr == t:
                    rp -= wrap
                    tr += W
                copies.append(rp)
                rp += stride

        def next_event(t):
            return max(min(max(min(tw, tr - PF), 0) & ~(GS - 1), tail), t)

        for s in range(PF):
            copy_step(s)
        te = next_event(0)
        t = 0
        while t < n:
            if t < te:
                assert t + PF + GS - 1 < n
                for _ in range(GS):
                    copies.append(rp)
                    rp += stride
                    stores.append(wp)
                    wp += stride
            else:
                for u in range(GS):
                    copy_step(t + PF + u)
                for u in range(GS):
                    if t + u < n:
                        if tw == t + u:
                            restarts.append(base + t + u)
                            wp -= wrap
                            tw += W
                        stores.append(wp)
                        wp += stride
                te = next_event(t + GS)
            t += GS
        tw -= 0 if tw == NEVER else n
        base += n
    return copies, stores, restarts


def _long_walk(W, H, kind, j, paired, G):
    """The same of the walk with one chain per warp: chunks of G steps, one cursor per step."""
    sh = 0 if kind < 2 else (1 if kind < 4 else -1)
    back = kind & 1
    dy, dx = (-1, -sh) if back else (1, sh)
    ystart = H - 1 if back else 0
    x = (j + sh * ystart) % W
    stride, wrap = dy * W + dx, dx * W
    wo = ystart * W + x

    def wrapped(xx, o):
        return (xx - dx * W, o - wrap) if xx >= W or xx < 0 else (xx, o)

    copies, stores, restarts = [], [], []
    fresh, base = False, 0
    for ph in range(2 if paired else 1):
        n = H if not paired else (H // 2 if (ph == 0) != bool(back) else H - H // 2)
        cur = [wrapped(x + dx * u, wo + u * stride) for u in range(G)]
        for k in range((n + G - 1) // G):
            for u in range(G):
                if k * G + u < n:
                    copies.append(cur[u][1])
                cur[u] = wrapped(cur[u][0] + G * dx, cur[u][1] + G * stride)
        for k in range((n + G - 1) // G):
            m, last = min(G, n - k * G), x + G * dx
            if m == G and not fresh and 0 <= last < W:
                stores += [wo + u * stride for u in range(G)]
                wo, x = wo + G * stride, last
            else:
                for u in range(m):
                    if fresh:
                        restarts.append(base + k * G + u)
                    stores.append(wo)
                    wo, x = wo + stride, x + dx
                    fresh = x >= W or x < 0
                    x, wo = wrapped(x, wo)
        base += n
    return copies, stores, restarts


@pytest.mark.parametrize("kind", range(6))
def test_sheared_walk_on_planes(host, kind):
    _, G, ring, GS, PF = host["const"][()]
    assert ring & (ring - 1) == 0 and GS + PF <= ring
    for W, H in itertools.product((1, 2, 3, 5, 8, 13, 40), (1, 2, 5, 6, 7, 8, 9, 14, 15, 33, 100)):
        sh = 0 if kind < 2 else (1 if kind < 4 else -1)
        for j in range(W):
            rows = range(H - 1, -1, -1) if kind & 1 else range(H)
            want = [y * W + (j + sh * y) % W for y in rows]
            entry = (0 if sh > 0 else W - 1) if not kind & 1 else (W - 1 if sh > 0 else 0)
            starts = [t for t, p in enumerate(want) if sh and t and p % W == entry]
            for paired in (False, True):
                got = _walk(W, H, kind, j, paired, GS, PF)
                assert got == (want, want, starts), (W, H, j, paired)
                if W >= G:
                    got = _long_walk(W, H, kind, j, paired, G)
                    assert got == (want, want, starts), (W, H, j, paired, "long")


@pytest.mark.parametrize("back", [False, True])
def test_row_walk_chunks(host, back):
    G = host["const"][()][1]
    for W, paired in itertools.product(range(1, 60), (False, True)):
        mid = host["mid"][(W,)]
        assert mid % G == 0
        got, met = [], [0, 0]
        for ph in range(2 if paired else 1):
            low = paired and (ph == 0) != back
            q0, q1 = (mid if paired and not low else 0), (mid if low else W)
            for k in range((q1 - q0 + G - 1) // G):
                n = min(G, q1 - q0 - k * G)
                p = q1 - k * G - n if back else q0 + k * G
                assert q0 <= p and p + n <= q1
                got += [p + (n - 1 - u if back else u) for u in range(n)]
            met[ph] = (q0, q1)
        assert got == (list(range(W - 1, -1, -1)) if back else list(range(W)))
        if paired:  # each part covers what the other direction covers in its other part
            assert met == ([(mid, W), (0, mid)] if back else [(0, mid), (mid, W)])


@pytest.mark.parametrize("W,D,T", [(1, 16, 32), (5, 32, 32), (37, 16, 32), (61, 48, 32),
                                   (80, 64, 64), (70, 256, 32)])
def test_selection_scans_every_sum_once(W, D, T):
    # each (pixel, d) with a target x - d >= 0 reaches that target exactly once, and nothing else
    # does; all word reads stay inside the tile
    h, pitch = D // 2, D // 2 + 1
    seen = {}
    for x0 in range(0, W, T):
        n = min(T, W - x0)
        for j in range(n + D - 1):
            t = j - (D - 1)
            if x0 + t < 0:
                continue
            par = t & 1
            assert (par - t) % 2 == 0
            kb, w = (par - t) // 2, par * pitch + (par - t) // 2
            for _ in range(par, T, 32):
                for i in range(16):
                    if 0 <= kb + i < h:
                        word = w + i * (2 * pitch + 1)
                        px, k = divmod(word, pitch)
                        assert 0 <= px < T and k == kb + i
                        if px < n:  # the other rows hold no sum
                            # low half d = 2k to target t, high half d = 2k + 1 to target t - 1
                            # (read by the target's thread from the next diagonal)
                            seen.setdefault((x0 + px, 2 * k), []).append(x0 + t)
                            if j >= 1 and x0 + t - 1 >= 0:
                                seen.setdefault((x0 + px, 2 * k + 1), []).append(x0 + t - 1)
                kb, w = kb + 16, w + 16 * (2 * pitch + 1)
    want = {(x, d): [x - d] for x in range(W) for d in range(min(D, x + 1))}
    assert seen == want


@pytest.mark.parametrize("D", range(16, 257, 16))
def test_ring_accesses_stay_inside(host, D):
    # shared-memory reads and copies of the row walk and of the walk with one chain per warp, in the
    # bytes planar_ring_smem gives one warp: costs and the other direction's U, stages of G pixels
    stages, G = host["const"][()][:2]
    assert stages & (stages - 1) == 0
    shapes = [(host["words"][(D,)], 32)]  # one chain per warp
    for dpl in (2, 4, 8):
        if (D, dpl) in host["lanes"]:
            shapes.append((dpl // 2, host["lanes"][(D, dpl)]))
    for nw, lpl in shapes:
        cpw = 32 // lpl
        assert 2 * nw * lpl >= D
        size = host["ring"][(D, lpl)]
        slot_bytes = cpw * G * D
        other = stages * slot_bytes
        for lane in range(32):
            c, lig = lane // lpl, lane % lpl
            at = host["at"][(D, nw, lig)]
            assert at == (lig * 2 * nw if lig * 2 * nw < D else 0)
            for stage in range(stages):
                base = c * G * D + stage * slot_bytes + other
                assert base + (G - 1) * D + at + 2 * nw <= size
                for v in range(nw):
                    i = lig + lpl * v
                    if i < G * D // 16:
                        assert base + 16 * i + 16 <= size
        # every piece of a chunk is copied by some lane
        assert {lig + lpl * v for lig in range(lpl) for v in range(nw)} >= set(range(G * D // 16))


def test_selection_tiles(host):
    # whole blocks of 32 pixels, no more than asked for, and the sums with the keys behind them
    for (D, T), (px, smem) in host["tile"].items():
        assert px % 32 == 0 and 32 <= px <= T
        assert smem == px * (D // 2 + 1) * 4 + (px + D) * 8 <= 32 * 1024


def test_shape_of_the_sheared_chains(host):
    # one chain per warp on small images whose rows are not the longer walk
    assert host["shape"] == {(160, 120, 8): 8, (320, 240, 8): 8, (320, 120, 8): 16,
                             (413, 307, 8): 16, (1000, 375, 4): 16, (640, 375, 4): 8,
                             (7, 9, 8): 16, (8, 9, 8): 8}
