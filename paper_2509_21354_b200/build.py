"""Build libkve.so (the CUDA library behind include/kve.h) in-tree with nvcc for sm_100a.

    python -m paper_2509_21354_b200.build [--force] [--verbose]
"""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libkve.so")
SOURCES = ["api.cu", "append.cu", "summarize.cu", "summarize_token.cu", "gate_rnn.cu", "gate_step.cu", "compact.cu", "attn.cu", "attn_block.cu", "attn_block_tc.cu", "attn_block_warp.cu", "selftest.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _deps_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [os.path.join(HERE, "..", "include", "kve.h")]
    return max(os.path.getmtime(f) for f in files)


def bind_path() -> str:
    """Where the decode step's extension module (csrc/bind.cpp) lies for this interpreter and this torch: it is compiled against
    the headers of both, and one that was built for others must not be loaded."""
    import hashlib
    import sysconfig
    import torch
    key = f"{sysconfig.get_config_var('SOABI')} {torch.__version__} {torch.version.cuda} {int(torch.compiled_with_cxx11_abi())}"
    return os.path.join(HERE, f"_kve_bind.{hashlib.sha256(key.encode()).hexdigest()[:12]}.so")


def build_bind(force: bool = False) -> str:
    """Compiles csrc/bind.cpp (an extension module against this interpreter and this torch; no device code)."""
    src, BIND = os.path.join(CSRC, "bind.cpp"), bind_path()
    if not force and os.path.exists(BIND) and os.path.getmtime(BIND) >= os.path.getmtime(src):
        return BIND
    import sysconfig
    import torch
    root = os.path.join(os.path.dirname(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    include = [sysconfig.get_paths()["include"], os.path.join(root, "include"),
               os.path.join(root, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    tmp = f"{BIND}.{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           *[f"-I{d}" for d in include], src, "-o", tmp, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stderr)
        raise RuntimeError("g++ failed on bind.cpp")
    os.replace(tmp, BIND)
    return BIND


def build(force: bool = False, verbose: bool = False, defines=(), lib: str = LIB, obj_dir: str = OBJ) -> str:
    """Compiles every source for sm_100a and links `lib`.  `defines` (e.g. ("KVE_ATTN_STAMPS",)) with another `lib`
    and `obj_dir` gives an instrumented copy beside the product library."""
    LIB, OBJ = lib, obj_dir
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    objs = []
    log = []
    for src in SOURCES:
        obj = os.path.join(OBJ, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, *[f"-D{d}" for d in defines], "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        log.append(r.stderr)
        if r.returncode != 0:
            sys.stderr.write(r.stderr)
            raise RuntimeError(f"nvcc failed on {src}")
        objs.append(obj)
    r = subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs],
                       capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stderr)
        raise RuntimeError("link failed")
    with open(os.path.join(OBJ, "ptxas.log"), "w") as f:
        f.write("\n".join(log))
    if verbose:
        print("\n".join(log))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
    print(build_bind(force="--force" in sys.argv))
