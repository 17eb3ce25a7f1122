"""Host-side logic of the launchers that needs neither a GPU nor the CUDA toolkit: compiled with g++ and run."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_per_device_setup_bookkeeping(tmp_path):
    exe = str(tmp_path / "device_once_check")
    src = os.path.join(ROOT, "tests", "host", "device_once_check.cpp")
    inc = os.path.join(ROOT, "paper_2503_02495_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip() == "ok"


def test_bound_on_the_weight_gradient_line(tmp_path):
    exe = str(tmp_path / "wgrad_line_check")
    src = os.path.join(ROOT, "tests", "host", "wgrad_line_check.cpp")
    inc = os.path.join(ROOT, "paper_2503_02495_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip() == "ok"


def test_setup_bookkeeping_under_threads(tmp_path):
    exe = str(tmp_path / "device_once_threads")
    src = os.path.join(ROOT, "tests", "host", "device_once_threads.cpp")
    inc = os.path.join(ROOT, "paper_2503_02495_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-Wall", "-Werror", "-pthread", "-fsanitize=thread", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip() == "ok"


def test_hand_over_between_warps_ends_in_every_order(tmp_path):
    exe = str(tmp_path / "hand_over_check")
    src = os.path.join(ROOT, "tests", "host", "hand_over_check.cpp")
    inc = os.path.join(ROOT, "paper_2503_02495_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip().endswith("ok")


def test_rules_of_launches(tmp_path):
    exe = str(tmp_path / "launch_rules_check")
    src = os.path.join(ROOT, "tests", "host", "launch_rules_check.cpp")
    inc = os.path.join(ROOT, "paper_2503_02495_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip() == "ok"
