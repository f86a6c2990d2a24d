"""The FFN kernels' work walk, the code the kernels compile, on host threads (walk_host.cc; CPU
only): every (segment, tile, k chunk) of the routed and the shared experts' work is walked exactly
once, by single CTAs and by pairs, and nothing the lanes and roles hand to one another relies on
less than the synchronisation that stands between them."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _build(out, *flags):
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-fno-strict-aliasing",
           "-I", os.path.join(ROOT, "paper_2505_19645_b200", "csrc"), *flags,
           os.path.join(HERE, "walk_host.cc"), "-o", str(out), "-lpthread"]
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
    exe = _build(tmp_path / "walk_tsan", "-fsanitize=thread")
    r = subprocess.run([exe, "2", "40"], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, TSAN_OPTIONS="halt_on_error=1"))
    assert "data race" not in r.stderr, r.stderr[:3000]
    assert r.returncode == 0 and "walks agree" in r.stdout, r.stdout + r.stderr[-2000:]
