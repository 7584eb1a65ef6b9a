"""Per-group products: when a wait gives up, the watching warp and the epilogue warps leave behind the same tile. No named barrier
keeps a part of its warps, and a CTA is through within two limits however many tiles are left. Every order of the steps of a small
CTA is gone through here; the sources are held to the steps gone through; on the GPU a wait is made to run out."""
import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")
CSRC = os.path.join(ROOT, "paper_2312_05693_b200", "csrc")
STAGES = 2                     # accumulator stages


def outcome(verdict, warps, tiles, blocks, issued, watcher_waits=True):
    """All orders of one watcher and `warps` epilogue warps of a lane quarter when MMAs stop after `issued` blocks. Returns the bad
    ends: a step that no other one can release ("stuck"), a wait for a release that never comes ("late").
    verdict "watcher": the watcher's word names the tile. "flag": every warp looks at the flag for itself.
    The warps start when the kernel ahead has completed; a wait for their releases may run out before that, not after.
    watcher_waits: the watcher, too, arrives for blocks that never came only then (others have not come before)."""
    total = tiles * blocks
    # (block, live, word) of the watcher; per warp (block, state: 0 arrive, 1 blocked, 2 release, 3 tile's end, 4 left); arrivals at
    # a barrier per stage; releases per block; whether the flag is up; whether the kernel ahead has completed
    start = (0, True, -1, tuple((0, 0) for _ in range(warps)), (0,) * STAGES, (0,) * total, False, False)
    seen, todo, bad = {start}, [start], set()

    def stage(b):
        return b % blocks % STAGES

    def before(b):                                     # the block that used b's stage last
        return max((c for c in range(b) if stage(c) == stage(b)), default=None)

    def arrive(ws, bars, s):
        bars = list(bars)
        bars[s] += 1
        if bars[s] == warps + 1:
            bars[s] = 0
            ws = [(b, 2) if st == 1 and stage(b) == s else (b, st) for b, st in ws]
        return tuple(ws), tuple(bars)

    while todo:
        state = todo.pop()
        w, live, word, ws, bars, rel, flag, ahead = state
        nxt = []
        if not flag and issued < total:
            nxt.append((w, live, word, ws, bars, rel, True, ahead))
        if not ahead:
            nxt.append((w, live, word, ws, bars, rel, flag, True))
        watching = w < total and not (verdict == "watcher" and not live and w % blocks == 0 and w // blocks != word and word >= 0)
        if watching and (ahead or not watcher_waits):
            prev = before(w)
            reusable = prev is None or rel[prev] == warps or not (live or ahead)
            came = live and w < issued and reusable
            if came or (not live and reusable) or (live and flag and reusable):
                ok = came
                nw = word
                if not ok and verdict == "watcher" and w % blocks == blocks - 1:
                    nw = w // blocks
                a, b = arrive(ws, bars, stage(w))
                nxt.append((w + 1, ok, nw, a, b, rel, flag, ahead))
            if not live and not reusable and all(st == 4 or (b, st) == (w, 1) for b, st in ws):
                bad.add("late")
        for i, (b, st) in enumerate(ws if ahead else ()):
            put = lambda v, ws=ws, i=i: tuple(v if j == i else x for j, x in enumerate(ws))
            if st == 0 and b < total:
                a, bb = arrive(list(put((b, 1))), bars, stage(b))
                nxt.append((w, live, word, a, bb, rel, flag, ahead))
            elif st == 2:
                r = list(rel)
                r[b] += 1
                nxt.append((w, live, word, put((b, 3) if b % blocks == blocks - 1 else (b + 1, 0)), bars, tuple(r), flag, ahead))
            elif st == 3:
                leave = word == b // blocks if verdict == "watcher" else flag
                nxt.append((w, live, word, put((b, 4) if leave or b + 1 == total else (b + 1, 0)), bars, rel, flag, ahead))
        if not nxt and (watching or any(st != 4 for _, st in ws)):
            bad.add("stuck")
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    return bad


@pytest.mark.parametrize("warps", [2, 3])
@pytest.mark.parametrize("tiles,blocks", [(1, 3), (2, 1), (3, 1), (2, 2), (2, 3), (3, 2)])
def test_every_order_ends(warps, tiles, blocks):
    for issued in range(tiles * blocks + 1):
        assert not outcome("watcher", warps, tiles, blocks, issued)


def test_a_look_at_the_flag_of_its_own_is_found_out():
    assert outcome("flag", 2, 2, 3, 1) >= {"stuck", "late"}


def test_a_watcher_ahead_of_its_warps_is_found_out():
    assert "stuck" in outcome("watcher", 2, 1, 6, 0, watcher_waits=False)


def test_the_kernel_takes_these_steps():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "aq_gemm_tensor.cu")).read())
    watcher = src[src.index("if (GROUPED && warp == 3)"):src.index("if (warp == 1 && elect_one())")]
    assert re.search(r"for \(int tl = 0; tl < my_tiles && live; \+\+tl\)", watcher)
    given_up = watcher[watcher.index("if (!live) {"):]
    assert given_up.index("griddepcontrol.wait") < given_up.index("drain_wait(") < given_up.index("sm.given_up = tl") < given_up.index("tell(a)")
    assert watcher.count("bar.arrive") == 1 and watcher.count("tell(a)") == 2
    epilogue = src[src.index("auto block = [&]"):src.index("role_done:")]
    assert "abort_flag" not in epilogue and "sm.given_up == tl" in epilogue


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,given_up", [(64, 4096, 128 * 444, 128 * 444),     # three tiles a CTA, of 64 tokens
                                            (100, 4096, 128 * 444, 128 * 444),    # of 128
                                            (192, 4096, 128 * 444, 128 * 444),    # of 192
                                            (192, 4096, 128 * 150, 128 * 148),    # shared tiles, in a launch of its own, behind a round
                                            (48, 4096, 1024, 0)])                 # in clusters, whose other CTAs may write outputs
def test_a_wait_that_runs_out_ends_the_call(M, K, N, given_up, tmp_path):
    import torch
    from gpu_util import handle
    from paper_2312_05693_b200 import binding
    h = handle()                                                   # the library is loaded
    lib = tmp_path / "starved_product.so"
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17",
                           "-shared", "-Xcompiler", "-fPIC", os.path.join(ROOT, "tests", "starved_product.cu"), "-o", str(lib),
                           "-L" + os.path.join(ROOT, "paper_2312_05693_b200"), "-l:libagileq.so",
                           "-Xlinker", "-rpath=" + os.path.abspath(os.path.join(ROOT, "paper_2312_05693_b200"))])
    fn = ctypes.CDLL(str(lib)).starved_product
    codes = torch.ones((M, K), dtype=torch.int8, device="cuda")
    packed = torch.zeros(binding.aq_packed_w4_bytes(N, K), dtype=torch.uint8, device="cuda")
    scales = torch.ones(binding.aq_scales_bytes(N, K, 128) // 2, dtype=torch.float16, device="cuda")
    y = torch.full((M, N), 7.0, dtype=torch.float16, device="cuda")
    ctl = torch.zeros(256, dtype=torch.uint8, device="cuda")
    scratch = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    ms = ctypes.c_float()
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (codes, packed, scales, y, ctl, scratch)]
    def call(busy, limit):
        ctl.zero_()
        y.fill_(7.0)
        torch.cuda.synchronize()
        assert fn(0, M, K, N, *ptr, ctypes.c_size_t(scratch.numel()), ctypes.c_ulonglong(busy), ctypes.c_ulonglong(limit), ctypes.byref(ms)) == 0
        return h.aq_check_workspace(ctl)

    for _ in range(2):
        assert call(1000, 4000000000) == binding.AQ_OK             # with time to spare (and the kernels loaded)
        assert bool((y == 0.0).all())
        # a limit of 20 ms at the highest clock, 65 ms at 600 MHz: it runs out while the kernel ahead still has most of its 300 ms
        assert call(300_000_000, 39_000_000) == binding.AQ_ERR_DEVICE_TIMEOUT, ms.value
        assert int(ctl[8:12].view(torch.int32).item()) in (1, 2, 3, 6, 7, 9)
        # no output of a tile that was given up; a CTA that only found its place behind the busy kernel has written its tiles
        tiles = (y[:, :given_up] == 7.0).reshape(M, -1, 128).sum((0, 2))
        assert bool(((tiles == 0) | (tiles == M * 128)).all()) and int((tiles == 0).sum()) <= given_up // 128 // 16
        assert ms.value < 300 + 2 * 65 + 50, ms.value              # a limit per block left would be 640 ms more at the least
