"""In-tree build of the C-ABI CUDA library (sm_100a) with nvcc.

`build_library()` compiles every `csrc/*.cu` to an object file and links `liblime_b200.so` next to this file; it needs nvcc and
nothing else.  `build_binding()` makes `_torch_binding.so` beside it, the native half of `binding.py` (`csrc/torch_binding.cpp`, host
code only); it needs g++, torch and Python's headers.  `build()` does both, and without what the second needs the library alone:
`binding.py` then marshals its calls in Python.  Objects are rebuilt only when a source or header is newer, the binding also when
torch or Python have changed.  nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import shutil
import subprocess
import sys
import sysconfig
from typing import Optional

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "liblime_b200.so")
BINDING = os.path.join(HERE, "_torch_binding.so")
MADE_FOR = os.path.join(OBJ, "torch_binding.made_for")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; the CUDA toolkit is required to build liblime_b200.so")
    return cand


def _newest(paths) -> float:
    return max(os.path.getmtime(p) for p in paths)


def binding_made_for() -> str:
    """The torch and the Python whose binary interfaces `_torch_binding.so` is compiled against."""
    import torch
    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def build_binding() -> Optional[str]:
    """The path of the extension, or None where something that it needs is not installed (said on stderr)."""
    src = os.path.join(CSRC, "torch_binding.cpp")
    try:
        made_for = binding_made_for()
        import torch
    except ImportError:
        made_for = None
    include = sysconfig.get_paths()["include"]
    missing = [what for what, there in (("torch", made_for is not None), ("g++", shutil.which("g++") is not None),
                                        ("Python.h", os.path.exists(os.path.join(include, "Python.h")))) if not there]
    if missing:
        print(f"[build] {', '.join(missing)} not found: _torch_binding.so is left out, binding.py marshals its calls in Python", file=sys.stderr)
        return None
    needs = [src, os.path.join(ROOT, "include", "lime.h"), __file__]
    if os.path.exists(BINDING) and os.path.getmtime(BINDING) >= _newest(needs) and os.path.exists(MADE_FOR) and open(MADE_FOR).read() == made_for:
        return BINDING
    home = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    includes = [os.path.join(ROOT, "include"), include, os.path.join(home, "include"),
                os.path.join(home, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f'-DLIME_MADE_FOR="{made_for}"',
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", src, "-o", BINDING]
    cmd += [f"-I{i}" for i in includes] + [f"-L{os.path.join(home, 'lib')}", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("g++ failed on " + src)
    os.makedirs(OBJ, exist_ok=True)
    with open(MADE_FOR, "w") as f:
        f.write(made_for)
    return BINDING


def build_library(verbose: bool = False, ptxas_info: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h")) + [__file__]
    hdr_time = _newest(headers)
    nvcc = _nvcc()
    jobs = []
    for src in sources:
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        if ptxas_info or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time):
            cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if ptxas_info else []) + ["-c", src, "-o", obj]
            jobs.append((src, cmd))

    def run(job):
        src, cmd = job
        r = subprocess.run(cmd, capture_output=True, text=True)
        return src, r

    with concurrent.futures.ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        for src, r in ex.map(run, jobs):
            if verbose or ptxas_info or r.returncode != 0:
                sys.stderr.write(f"[nvcc] {os.path.basename(src)}\n{r.stdout}{r.stderr}\n")
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}")
    objs = [os.path.join(OBJ, os.path.basename(s)[:-3] + ".o") for s in sources]
    if jobs or not os.path.exists(LIB) or os.path.getmtime(LIB) < _newest(objs):
        cmd = [nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    return LIB


def build(verbose: bool = False, ptxas_info: bool = False) -> str:
    lib = build_library(verbose, ptxas_info)
    build_binding()
    return lib


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, ptxas_info="--ptxas" in sys.argv))
