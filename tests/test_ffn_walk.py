"""The FFN kernels' work walk and rings, the code the kernels compile, on the host (CPU only).

walk_host.cc: every (segment, tile, k chunk) of the routed and the shared experts' work is walked exactly
once, by single CTAs and by pairs, and nothing the lanes and roles hand to one another relies on
less than the synchronisation that stands between them.  ring_host.cc: the token ring, the weight
slots and the k-step barriers in every geometry the host's rule gives.  tile_host.cc: the tile heights
the host gives the GPU tests' cases and others."""
import os
import random
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
        ctas, up, down, _ = map(int, line.split())
        cut = lambda rows, h: [min(h * ctas, rows - f) // ctas for f in range(0, rows, h * ctas)]  # noqa: E731
        out.append((ctas, cut(I, up), cut(H, down)))
    return out


# rows per CTA of the gate/up and the down tiles of the fixed cases of test_gpu_layer.py, on pairs in
# either ring geometry
PAIR_TILES = {
    "pair-tile-edges": ([64, 64, 48], [128, 16]),
    "pair-few-rows": ([64, 48], [80]),
    "pair-segments": ([64, 64, 64, 64, 16], [128]),
    "pair-half-box": ([48], [128, 128, 16]),
    "pair-mid-piece": ([64, 64, 16], [48]),
    "pair-tile-edges-full": ([128, 48], [144]),
    "pair-few-rows-full": ([112], [80]),
    "pair-segments-full": ([128, 128, 16], [128]),
    "pair-half-box-full": ([48], [256, 256, 16]),
    "pair-mid-piece-full": ([128, 128, 16], [48]),
    "rr-segments": ([64, 64, 64], [128]),
    "rr-ragged": ([64, 48], [80]),
    "rr-segments-full": ([128, 64], [128]),
    "rr-ragged-full": ([112], [80]),
    "rr-blocks-full": ([128, 48], [208]),
}
# the same on single CTAs (calls of up to 128 tokens, the host's own choice)
SINGLE_TILES = {
    "rr-ragged": ([64, 64, 64, 32], [128, 32]),
    "rr-ragged-full": ([128, 96], [160]),
    "rr-blocks-full": ([128, 128, 96], [256, 160]),
}


def test_gpu_cases_run_at_the_tile_heights_they_name(tmp_path):
    """The height of a routed tile follows from the number of items, so a case reaches an edge of a
    full-height tile, or of a cut one, only at the right number of groups."""
    from test_gpu_idle_tiles import IDLE_TILE_CASES
    from test_gpu_layer import PAIR_CASES, SCHEDULING_CASES
    from test_gpu_random_shapes import FULL_TILE_CASES, draw_full_tile_case

    exe = _build(tmp_path / "tile", "tile_host.cc")
    cases = {n: (H, E, k, I, Is, B * (g + 1)) for n, H, E, k, I, Is, B, g in PAIR_CASES + SCHEDULING_CASES}
    for wide in (0, 1):
        got = _tiles(exe, [cases[n] + (wide, 1) for n in PAIR_TILES])
        assert {n: (2, *t) for n, t in PAIR_TILES.items()} == dict(zip(PAIR_TILES, got))
    got = _tiles(exe, [cases[n] + (-1, 0) for n in SINGLE_TILES])
    assert {n: (1, *t) for n, t in SINGLE_TILES.items()} == dict(zip(SINGLE_TILES, got))

    # low tiles in both passes, in one of them
    idle = _tiles(exe, [c + (-1, 0) for c in IDLE_TILE_CASES if c[3] < 2048])
    assert all(max(up) <= 64 and max(down) <= 128 for _, up, down in idle[:-2])
    assert idle[-2:] == [(1, [128, 32], [128] * 4 + [32]), (2, [48], [256, 144])]

    # full tiles of the random shapes: ragged second down blocks, ragged gate/up tiles
    rng = random.Random(15)
    full = _tiles(exe, [draw_full_tile_case(rng) + (-1, 0) for _ in range(FULL_TILE_CASES)])
    second = [ctas for ctas, _, down in full if any(128 < h < 256 for h in down)]
    partial = [ctas for ctas, up, _ in full if any(64 < h < 128 for h in up)]
    assert len(second) >= 40 and second.count(2) >= 10, (len(second), second.count(2))
    assert len(partial) >= 40 and partial.count(2) >= 10, (len(partial), partial.count(2))


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


def test_a_small_gather_leaves_sms_to_the_shared_expert(tmp_path):
    """Up to 16 MB of rows the gather of a layer with a shared expert runs as one CTA per SM."""
    calls = {(512, 16, 4, 256, 512, 2080): 1, (512, 16, 4, 256, 512, 4096): 1, (512, 16, 4, 256, 512, 4097): 8,
             (512, 16, 4, 256, 0, 2080): 8, (7168, 256, 8, 2048, 2048, 3072): 8}
    lines = ["%d %d %d %d %d %d -1 0" % (E, k, H, I, Is, T) for H, E, k, I, Is, T in calls]
    r = subprocess.run([_build(tmp_path / "tile", "tile_host.cc")], input="\n".join(lines) + "\n",
                       capture_output=True, text=True, check=True)
    assert [int(v.split()[3]) for v in r.stdout.splitlines()] == list(calls.values())
