"""Build libag.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _marshal.so (its Python
argument marshalling) with the host compiler."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libag.so")
MARSHAL = os.path.join(HERE, "_marshal.so")
SOURCES = ["ag_api.cu", "gate.cu", "gemm_tc.cu", "gate_attn_tc.cu", "gate_linear.cu", "compact.cu", "prefill.cu", "prefill_tc.cu", "decode.cu", "decode_gqa_mma.cu", "kv_proj_cache.cu", "out_proj.cu"]
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
NVCC_FLAGS = [*ARCH, "-lineinfo", "-O3", "-std=c++17", "--use_fast_math", "-Xcompiler", "-fPIC",
              "-cudart", "static"]


def _newest_source_mtime():
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    paths.append(os.path.join(HERE, "..", "include", "ag.h"))
    paths.append(os.path.abspath(__file__))
    return max(os.path.getmtime(p) for p in paths)


def marshal_tag():
    """What _marshal.so depends on beside its sources: it reads torch's tensors and Python's objects by their layout."""
    import sysconfig
    import torch
    return f"AG_MARSHAL_FOR torch {torch.__version__} python {sysconfig.get_config_var('SOABI')}"


def marshal_matches(path):
    """Whether the module at `path` was built for this torch and this Python; its tag lies in it as text."""
    with open(path, "rb") as f:
        return marshal_tag().encode() + b"\0" in f.read()


def build_marshal(force=False):
    """Compile csrc/py_binding.cpp into _marshal.so, linked against libag.so and torch."""
    src = os.path.join(CSRC, "py_binding.cpp")
    newest = max(os.path.getmtime(p) for p in (src, os.path.join(HERE, "..", "include", "ag.h"), os.path.abspath(__file__)))
    if not force and os.path.exists(MARSHAL) and os.path.getmtime(MARSHAL) >= newest and marshal_matches(MARSHAL):
        return MARSHAL
    import sysconfig
    import torch
    T = os.path.join(os.path.dirname(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    inc = [os.path.join(T, "include"), os.path.join(T, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    # torch's own libraries are in the process already when the module is imported; libag.so lies beside it
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
                    f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DAG_MARSHAL_TAG="{marshal_tag()}"',
                    *[f"-I{p}" for p in inc], src, "-o", MARSHAL, f"-L{HERE}", "-lag", "-Wl,-rpath,$ORIGIN",
                    "-L" + os.path.join(T, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"], check=True)
    return MARSHAL


def build(force=False, verbose=False):
    """Compile every .cu under csrc/ into libag.so, and _marshal.so; returns the library path."""
    build_lib(force, verbose)
    build_marshal(force)
    return LIB


def build_lib(force=False, verbose=False):
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs, procs = [], []
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    for src in SOURCES:
        obj = os.path.join(HERE, "_build", src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip():
            print(f"--- {src}\n{out}", file=sys.stderr)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.run([nvcc, "-shared", "-cudart", "static", *ARCH, "-o", LIB, *objs], check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
