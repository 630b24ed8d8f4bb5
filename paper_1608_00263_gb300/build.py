"""Builds the CUDA library ``libqs.so`` in-tree for sm_103a.

Each translation unit under ``csrc/`` is compiled in parallel with nvcc
(``-gencode arch=compute_103a,code=sm_103a -lineinfo -O3``), then linked
into ``paper_1608_00263_gb300/libqs.so``.  Objects go to ``_build/``.
``build(checked=True)`` makes the checked build ``libqs_checked.so``
(``-DQS_CHECKED``: device-side index checks, objects in ``_build_checked/``),
which the binding loads when the environment sets ``QS_CHECKED=1``.
Host code carries no architecture-specific flags, so the same sources build
on x86_64 and aarch64 hosts.
"""
import concurrent.futures as cf
import hashlib
import importlib.util
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libqs.so")
BUILD_CHECKED = os.path.join(PKG, "_build_checked")
LIB_CHECKED = os.path.join(PKG, "libqs_checked.so")
GENCODE = "arch=compute_103a,code=sm_103a"


def _nvcc():
    cand = [os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"]
    for c in cand:
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC)
                  if f.endswith((".cu", ".cpp")))


def _headers():
    hs = [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith((".h", ".cuh", ".inc", ".py"))]
    hs.append(os.path.join(ROOT, "include", "qs.h"))
    return hs


def _flags(checked=False):
    common = ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include")]
    return common + ["-gencode", GENCODE, "-lineinfo"] + (["-DQS_CHECKED"] if checked else [])


def _generate(build_dir):
    """Writes the generated sources (the wide pass's op loop, the statistics'
    logarithm table) into the build directory."""
    for name in ("op_loop", "log_table"):
        spec = importlib.util.spec_from_file_location("gen_" + name, os.path.join(CSRC, "gen_%s.py" % name))
        gen = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(gen)
        with open(os.path.join(build_dir, "qs_%s.inc" % name), "w") as f:
            f.write(gen.emit())


def _digest(paths, extra):
    h = hashlib.sha1()
    for p in paths:
        with open(p, "rb") as f:
            h.update(f.read())
    h.update(" ".join(extra).encode())
    return h.hexdigest()


def _compile(nvcc, src, flags, verbose, build_dir=BUILD):
    obj = os.path.join(build_dir, os.path.basename(src) + ".o")
    cmd = [nvcc] + flags + ["-c", src, "-o", obj]
    if verbose and src.endswith(".cu"):
        cmd += ["-Xptxas", "-v"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
    return obj, r.stderr


def build(force=False, verbose=False, checked=False):
    nvcc = _nvcc()
    build_dir, lib = (BUILD_CHECKED, LIB_CHECKED) if checked else (BUILD, LIB)
    os.makedirs(build_dir, exist_ok=True)
    srcs = _sources()
    flags = _flags(checked)
    digest = _digest(srcs + _headers(), flags + [nvcc, sys.platform, os.uname().machine])
    stamp = os.path.join(build_dir, "stamp")
    if not force and os.path.exists(lib) and os.path.exists(stamp):
        with open(stamp) as f:
            if f.read().strip() == digest:
                return lib
    _generate(build_dir)
    flags = flags + ["-I" + build_dir]
    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        results = list(ex.map(lambda s: _compile(nvcc, s, flags, verbose, build_dir), srcs))
    if verbose:
        for _, err in results:
            if err:
                sys.stderr.write(err)
    tmp = lib + ".tmp%d" % os.getpid()
    cmd = [nvcc, "-shared", "-gencode", GENCODE, "-o", tmp] + [o for o, _ in results] + ["-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, lib)
    with open(stamp, "w") as f:
        f.write(digest)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, checked="--checked" in sys.argv))
