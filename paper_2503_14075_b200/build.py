"""Builds the C-ABI shared library (libtwig.so) in-tree with nvcc for sm_100a, and the native module
of the Python binding (_binding) with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.environ.get("TWIG_LIB") or os.path.join(HERE, "libtwig.so")   # TWIG_LIB: load another build
SOURCES = ["api.cu", "ttp.cu", "ttp_mq.cu", "tree_attn.cu", "tensor_maps.cu", "tree_attn_narrow.cu", "tree_attn_wide.cu", "tree_attn_stream.cu", "tree_accept.cu", "tree_build.cu", "chain_draft.cu"]


BINDING = os.path.join(HERE, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))


def _newest_source_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(ROOT, "include", "twig.h"))
    return max(os.path.getmtime(f) for f in files)


def is_stale() -> bool:
    newest = _newest_source_mtime()
    return any(not os.path.exists(f) or os.path.getmtime(f) < newest for f in (LIB, BINDING))


def _run(cmd, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{os.path.basename(cmd[0])} failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stderr)


def _build_binding(verbose: bool) -> None:
    import torch
    base = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    include = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), os.path.join(ROOT, "include"), sysconfig.get_path("include")]
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", *("-I" + d for d in include),
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", os.path.join(CSRC, "binding.cpp"),
          "-L" + os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda",
          "-o", BINDING], verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    arch = ["-gencode", "arch=compute_100a,code=sm_100a"]
    flags = arch + ["-O3", "-std=c++17", "-lineinfo", "-DTWIG_BUILD", "-Xcompiler", "-fPIC,-O2",
                    "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]
    # one compiler process per source file
    with tempfile.TemporaryDirectory() as tmp, ThreadPoolExecutor(os.cpu_count() or 1) as pool:
        objects = [os.path.join(tmp, os.path.splitext(s)[0] + ".o") for s in SOURCES]
        jobs = [pool.submit(_run, [nvcc, *flags, "-c", os.path.join(CSRC, s), "-o", o], verbose)
                for s, o in zip(SOURCES, objects)]
        jobs.append(pool.submit(_build_binding, verbose))
        for job in jobs:
            job.result()
        _run([nvcc, *arch, "-shared", "-Xcompiler", "-fPIC", "-o", LIB, *objects], verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
