"""Compile the CUDA sources in ``csrc/`` into ``libqnn_b200.so`` (sm_100a only), and
``csrc/fastcall.c`` into the extension module the binding makes its calls through.

nvcc cross-compiles without a GPU.  Objects are rebuilt only when their source
(or a header) is newer; translation units compile in parallel.
"""
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
OBJ_DIR = os.path.join(_HERE, "_build")
LIB = os.path.join(_HERE, "libqnn_b200.so")
# the binding's host path (csrc/fastcall.c); the name carries the interpreter's ABI, so that no other one loads it
FASTCALL = os.path.join(_HERE, "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
]


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers_mtime():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return max(os.path.getmtime(h) for h in hs)


def _compile(src, verbose):
    obj = os.path.join(OBJ_DIR, src[:-3] + ".o")
    cmd = ["nvcc", "-c", os.path.join(CSRC, src), "-o", obj] + NVCC_FLAGS
    if verbose:
        cmd += ["-Xptxas", "-v"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    return obj, r.stderr


def _build_fastcall(force: bool = False) -> bool:
    """The extension module, if there is a C compiler and the interpreter's headers; without it the binding
    makes the same calls through ctypes."""
    src = os.path.join(CSRC, "fastcall.c")
    if not force and os.path.exists(FASTCALL) and os.path.getmtime(FASTCALL) >= os.path.getmtime(src):
        return True
    # what stands there was made from another source, or (without a tag) perhaps for another interpreter
    for old in (FASTCALL, os.path.join(os.path.dirname(FASTCALL), "_fastcall.so")):
        if os.path.exists(old):
            os.remove(old)
    cmd = ["gcc", "-O2", "-shared", "-fPIC", "-Wall", "-I", sysconfig.get_paths()["include"], src, "-o", FASTCALL]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
        built, log = r.returncode == 0, r.stderr
    except OSError as e:
        built, log = False, str(e)
    if not built:
        print(f"{os.path.basename(FASTCALL)} not built, calls go through ctypes:\n{log}", file=sys.stderr)
    return built


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ_DIR, exist_ok=True)
    hm = _headers_mtime()
    todo, objs = [], []
    for src in _sources():
        obj = os.path.join(OBJ_DIR, src[:-3] + ".o")
        objs.append(obj)
        sm = max(os.path.getmtime(os.path.join(CSRC, src)), hm)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < sm:
            todo.append(src)
    if todo:
        with ThreadPoolExecutor(max_workers=min(8, len(todo))) as ex:
            for obj, log in ex.map(lambda s: _compile(s, verbose), todo):
                if verbose:
                    sys.stderr.write(log)
    if todo or not os.path.exists(LIB):
        cmd = ["nvcc", "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        subprocess.run(cmd, check=True)
    _build_fastcall(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
