"""Build libcomfuse.so (sm_100a only) from csrc/*.cu with nvcc, in-tree.

    python -m paper_2608_03537_b200.build [--force] [--verbose] [--checked]

--checked builds paper_2608_03537_b200/libcomfuse_checked.so (objects under build/obj_checked) with -DCOMFUSE_CHECKED: the
kernels' bounds predicates are compiled in; a predicate that fails records COMFUSE_ERR_BOUNDS in the device status word and
the access is skipped.  COMFUSE_LIB=<path> makes the Python binding load that library instead of libcomfuse.so.

_binding.<Python's tag>.so (csrc/binding.c, the argument marshalling of the Python entry points) is built beside the library, with
the C compiler ($CC, else gcc) and the headers of the Python that runs this; another Python version does not load it.

Each translation unit is compiled in parallel to build/obj/*.o and linked into
paper_2608_03537_b200/libcomfuse.so.  A unit is rebuilt when it, or any header in
csrc/ or include/, is newer than its object.  The kernel headers are also embedded in the library as text
(build/gen/embedded_sources.cpp): stage programs are compiled against them at run time.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
OBJ_DIR = os.path.join(ROOT, "build", "obj")
LIB_PATH = os.path.join(PKG_DIR, "libcomfuse.so")
BINDING_PATH = os.path.join(PKG_DIR, "_binding" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC",
    "-I", os.path.join(ROOT, "include"),
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if os.path.exists(cand) else "nvcc"


def _newest_header_mtime() -> float:
    m = 0.0
    for d in (CSRC, os.path.join(ROOT, "include")):
        for f in os.listdir(d):
            if f.endswith((".h", ".cuh")):
                m = max(m, os.path.getmtime(os.path.join(d, f)))
    return m


# the kernel headers a stage program is compiled against at run time (csrc/compiled_program.cu), by #include name
EMBEDDED = [
    (os.path.join(ROOT, "include", "comfuse.h"), "comfuse.h"),
    (os.path.join(CSRC, "fused_params.h"), "fused_params.h"),
    (os.path.join(CSRC, "sm100_primitives.cuh"), "sm100_primitives.cuh"),
    (os.path.join(CSRC, "epilogue_common.cuh"), "epilogue_common.cuh"),
    (os.path.join(CSRC, "fused_pair.cuh"), "fused_pair.cuh"),
]


def _write_embedded_sources(gen_dir: str) -> str:
    """Writes the text of the EMBEDDED headers as string constants (one C++ file); rewritten only when it changes."""
    os.makedirs(gen_dir, exist_ok=True)
    out = ["// generated by build.py: kernel sources for run-time compilation", "namespace comfuse {"]
    names = []
    for i, (path, name) in enumerate(EMBEDDED):
        text = open(path).read()
        assert ')COMFUSE_SRC"' not in text
        out.append(f"static const char kSource{i}[] =")
        lines = text.splitlines(keepends=True)
        for j in range(0, len(lines), 100):   # raw string literals of 100 lines each, concatenated by the compiler
            out.append('R"COMFUSE_SRC(' + "".join(lines[j:j + 100]) + ')COMFUSE_SRC"')
        out.append(";")
        names.append(name)
    out.append("extern const char* const kEmbeddedSourceNames[] = {" + ", ".join(f'"{n}"' for n in names) + "};")
    out.append("extern const char* const kEmbeddedSources[] = {" + ", ".join(f"kSource{i}" for i in range(len(names))) + "};")
    out.append(f"extern const int kEmbeddedSourceCount = {len(names)};")
    out.append("}  // namespace comfuse")
    text = "\n".join(out) + "\n"
    path = os.path.join(gen_dir, "embedded_sources.cpp")
    if not os.path.exists(path) or open(path).read() != text:
        with open(path, "w") as f:
            f.write(text)
    return path


def _compile(src: str, obj: str, verbose: bool, checked: bool = False) -> None:
    cmd = [_nvcc(), *NVCC_FLAGS, "-c", src, "-o", obj]
    if checked:
        cmd.insert(1, "-DCOMFUSE_CHECKED")
    if os.environ.get("COMFUSE_BUILD_TRACE"):   # phase-timestamp tracing build (see fused_params.h: trace)
        cmd.insert(1, "-DCOMFUSE_TRACE")
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}")


def build_binding(force: bool = False) -> str:
    """The argument-marshalling extension of the Python entry points (host code, one C file)."""
    src = os.path.join(CSRC, "binding.c")
    newest = max(os.path.getmtime(src), os.path.getmtime(os.path.join(ROOT, "include", "comfuse.h")))
    untagged = os.path.join(PKG_DIR, "_binding.so")   # what a build once wrote: any Python version would load it
    if untagged != BINDING_PATH and os.path.exists(untagged):
        os.remove(untagged)
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")):
        raise RuntimeError(f"{include}/Python.h not found: the headers of this Python are needed to compile {src}")
    if force or not os.path.exists(BINDING_PATH) or os.path.getmtime(BINDING_PATH) < newest:
        cmd = [os.environ.get("CC") or "gcc", "-O2", "-shared", "-fPIC", "-std=c11", "-I", include, "-I", os.path.join(ROOT, "include"),
               src, "-o", BINDING_PATH]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError(f"compiling {src} failed")
    return BINDING_PATH


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    obj_dir = OBJ_DIR + "_checked" if checked else OBJ_DIR
    lib_path = os.path.join(PKG_DIR, "libcomfuse_checked.so") if checked else LIB_PATH
    os.makedirs(obj_dir, exist_ok=True)
    build_binding(force)
    sources = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
    hdr_m = _newest_header_mtime()
    jobs, objs = [], []
    for f in sources:
        src = os.path.join(CSRC, f)
        obj = os.path.join(obj_dir, f[:-3] + ".o")
        objs.append(obj)
        stale = force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_m)
        if stale:
            jobs.append((src, obj))
    emb = _write_embedded_sources(os.path.join(ROOT, "build", "gen"))
    emb_obj = os.path.join(obj_dir, "embedded_sources.o")
    objs.append(emb_obj)
    if force or not os.path.exists(emb_obj) or os.path.getmtime(emb_obj) < os.path.getmtime(emb):
        jobs.append((emb, emb_obj))
    if jobs:
        with ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            list(ex.map(lambda j: _compile(j[0], j[1], verbose, checked), jobs))
    if jobs or not os.path.exists(lib_path):
        cmd = [_nvcc(), "-shared", "-o", lib_path, *objs, "-gencode", "arch=compute_100a,code=sm_100a", "-ldl"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    return lib_path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, checked="--checked" in sys.argv))
