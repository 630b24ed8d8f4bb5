"""Shared memory of the persistent wide batch kernel between work items: the
kernel's text, compiled with one host thread per CUDA thread, all but the first
held up after every barrier (persistent_cta_model.cpp)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def kernel_text():
    with open(os.path.join(ROOT, "paper_1608_00263_gb300", "csrc", "qs_wide.cu")) as f:
        s = f.read()
    at = s.index("k_batch_persistent_wide(float2")
    sum_at = s.index("__device__ __forceinline__ double sum_slots")
    text = s[sum_at:s.index("\n}\n", sum_at) + 3] + s[s.rindex("template <", 0, at):s.index("\n}\n", at) + 3]
    dyn = "extern __shared__ __align__(16) unsigned char smem_dyn[];"
    assert text.count(dyn) == 1
    return text.replace(dyn, "static unsigned char smem_dyn[16];")


def run_model(tmp_path, text):
    (tmp_path / "kernel.inc").write_text(text)
    exe = tmp_path / "model"
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I" + os.path.join(ROOT, "include"),
                    '-DKERNEL_TEXT="%s"' % (tmp_path / "kernel.inc"),
                    os.path.join(ROOT, "tests", "persistent_cta_model.cpp"),
                    os.path.join(ROOT, "paper_1608_00263_gb300", "csrc", "qs_host.cpp"), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)


def test_items_do_not_overlap(tmp_path):
    r = run_model(tmp_path, kernel_text())
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


@pytest.mark.parametrize("late", ["w.kind == kPersistStats", "barrier"])
def test_the_model_sees_a_late_read(tmp_path, late):
    """Planted: the item's kind read after the barrier that lets thread 0 go on
    to the next item; the closing barrier of a statistics item left out."""
    text = kernel_text()
    if late == "barrier":
        at = text.rindex("__syncthreads();")
        text = text[:at] + text[at + len("__syncthreads();"):]
        # (the threads that sum have to be late as well)
        text = text.replace("if (s_last &&", "if (late_read(s_last) &&")
        text = ("static int late_read(int &v) { if (threadIdx.x) std::this_thread::sleep_for("
                "std::chrono::milliseconds(5)); return v; }\n" + text)
    else:
        assert text.count("if (stats) {") == 2
        text = text.replace("if (stats) {", "if (w.kind == kPersistStats) {")
    # (several runs: on a busy host thread 0 may be held up too)
    for attempt in range(6):
        r = run_model(tmp_path, text)
        if r.returncode == 1:
            break
    assert r.returncode == 1 and r.stdout.strip(), r.stdout
