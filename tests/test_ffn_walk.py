"""The FFN kernels' work walk and rings, the code the kernels compile, on the host (CPU only).

walk_host.cc: every (segment, tile, k chunk) of the routed and the shared experts' work is walked exactly
once, by single CTAs and by pairs, and nothing the lanes and roles hand to one another relies on
less than the synchronisation that stands between them.  ring_host.cc: the token ring, the weight
slots and the k-step barriers in every geometry the host's rule gives."""
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
