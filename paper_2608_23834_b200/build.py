"""Builds libmkv.so (hand-written CUDA for sm_100a) and its Python binding in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmkv.so")
BINDING = os.path.join(HERE, "_mkv_native.so")     # marshalling of the Python calls (csrc/py_binding.cpp)
SOURCES = ["pool.cu", "lifecycle_kernels.cu", "decode_scalar.cu", "decode_tensor.cu", "decode_static.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = sources() + [os.path.join(CSRC, "py_binding.cpp"),
                        *(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")),
                        os.path.join(ROOT, "include", "mkv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def start_binding_object(obj):
    """Starts the host compiler on the Python binding, which sees tensors through PyTorch's C++ headers."""
    from torch.utils import cpp_extension
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], "/usr/local/cuda/include", os.path.join(ROOT, "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", *(a for i in inc for a in ("-isystem", i)), "-c",
           os.path.join(CSRC, "py_binding.cpp"), "-o", obj]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def link_binding(obj):
    # PyTorch's libraries are found among those that `import torch` has loaded; libmkv.so sits beside the binding
    from torch.utils import cpp_extension
    subprocess.run(["g++", "-shared", "-o", BINDING, obj, *(f"-L{p}" for p in cpp_extension.library_paths()), f"-L{HERE}",
                    "-l:libmkv.so", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"], check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    procs = []
    for src in sources():
        obj = os.path.join(HERE, "build", os.path.basename(src) + ".o")
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    binding_obj = os.path.join(HERE, "build", "py_binding.cpp.o")
    procs.append(("py_binding.cpp", start_binding_object(binding_obj)))
    log = []
    for src, p in procs:
        out, _ = p.communicate()
        log.append(out)
        if p.returncode != 0:
            sys.stderr.write(out)
            raise RuntimeError(f"the compiler failed on {src}")
    subprocess.run([nvcc, "-shared", "-o", LIB, *objs, "-lcudart"], check=True)
    link_binding(binding_obj)
    with open(os.path.join(HERE, "build", "ptxas.log"), "w") as f:
        f.write("\n".join(log))
    if verbose:
        print("\n".join(log))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
