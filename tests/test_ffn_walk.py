"""The FFN kernels' work walk and rings, the code the kernels compile, on the host (CPU only).

walk_host.cc: every (segment, tile, k chunk) of the routed and the shared experts' work is walked exactly
once, by single CTAs and by pairs, and nothing the lanes and roles hand to one another relies on
less than the synchronisation that stands between them.  ring_host.cc: the token ring, the weight
slots and the k-step barriers in every geometry the host's rule gives.  tile_host.cc: the tile heights
the host gives the GPU tests' cases and others."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _build(out, source="walk_host.cc", *flags):
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-fno-strict-aliasing", *flags,
           "-I", os.path.join(ROOT, "paper_2505_19645_b200", "csrc"), "-I", os.path.join(ROOT, "include"),
           os.path.join(HERE, source), "-o", str(out), "-lpthread"]
    subprocess.run(cmd, check=True)
    return str(out)


def test_every_piece_of_work_is_walked_exactly_once(tmp_path):
    r = subprocess.run([_build(tmp_path / "walk"), "1", "400"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "walks agree" in r.stdout, r.stdout + r.stderr


def test_no_hand_over_relies_on_less_than_it_waits_for(tmp_path):
    """Under ThreadSanitizer, where the stand-in for a warp vote orders no memory."""
    lib = subprocess.run(["g++", "-print-file-name=libtsan.so"], capture_output=True, text=True).stdout.strip()
    if not os.path.isabs(lib):
        pytest.skip("sanitizer run-time not installed")
    exe = _build(tmp_path / "walk_tsan", "walk_host.cc", "-fsanitize=thread")
    r = subprocess.run([exe, "2", "40"], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, TSAN_OPTIONS="halt_on_error=1"))
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("the sanitizer run-time does not fit this kernel's address space")
    assert "data race" not in r.stderr, r.stderr[:3000]
    assert r.returncode == 0 and "walks agree" in r.stdout, r.stdout + r.stderr[-2000:]


def test_rings_never_stall_and_never_reuse_what_is_live(tmp_path):
    r = subprocess.run([_build(tmp_path / "ring", "ring_host.cc"), "3", "60"], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "rings hold" in r.stdout, r.stdout + r.stderr
    # all three ring sizes, on single CTAs and on pairs, were among them
    assert all(int(v) > 0 for v in r.stdout.replace(",", "").replace(":", "").split() if v.isdigit()), r.stdout


def _tiles(exe, calls):
    """For calls (H, E, k, I, Is, T, MOE_FF_WIDE, MOE_FF_PAIR): CTAs per worker and the rows per CTA of
    a group's gate/up and down tiles."""
    lines = ["%d %d %d %d %d %d %d %d" % (E, k, H, I, Is, T, wide, pair)
             for H, E, k, I, Is, T, wide, pair in calls]
    r = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True)
    out = []
    for (H, _, _, I, *_), line in zip(calls, r.stdout.split("\n")):
        assert I < 2048   # (from there on the down pass may split its reduction)
        ctas, up, down = map(int, line.split())
        cut = lambda rows, h: [min(h * ctas, rows - f) // ctas for f in range(0, rows, h * ctas)]  # noqa: E731
        out.append((ctas, cut(I, up), cut(H, down)))
    return out


# (H, E, k, I, Is, T): rows per CTA of a tile in the two passes, where full height and low tiles were
# both timed; beside them the us per call at full height -> at this one -> at low tiles while each pass
# alone fits the SMs (64 rows in either).
MEASURED_HEIGHTS = {
    (256, 8, 2, 512, 0, 16): (64, 128),         # 18.3 -> 17.3 -> 17.4
    (512, 8, 2, 1024, 0, 16): (128, 128),       # 22.4 -> 21.0 -> 23.8
    (512, 16, 4, 512, 512, 16): (128, 128),     # 22.2 -> 21.3 -> 25.6
    (512, 16, 4, 512, 512, 160): (128, 128),    # 27.7 -> 26.8 -> 32.2
    (512, 64, 8, 256, 512, 5): (128, 256),      # 20.7 -> 20.7 -> 23.9
    (2048, 8, 2, 768, 1024, 160): (128, 256),   # 40.2 -> 40.2 -> 42.2
    (1024, 32, 2, 512, 512, 16): (128, 256),    # 27.2 -> 27.2 -> 27.2
}


def test_low_tiles_stand_where_they_were_faster(tmp_path):
    """Low tiles in the gate/up pass leave the down pass no SM to start on early, unless the items of
    both passes fit the SMs together."""
    got = _tiles(_build(tmp_path / "tile", "tile_host.cc"), [c + (-1, 0) for c in MEASURED_HEIGHTS])
    for (call, heights), (_, up, down) in zip(MEASURED_HEIGHTS.items(), got):
        assert (max(up), max(down)) == heights, call
