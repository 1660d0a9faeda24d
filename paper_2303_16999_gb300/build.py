"""Builds the native library ``_build/libspmm.so`` in-tree with nvcc.

Every CUDA source is compiled for sm_103a only
(``-gencode arch=compute_103a,code=sm_103a``), host C++ with the same nvcc
front end; translation units compile in parallel and are linked into one
shared library exporting the C ABI of ``include/spmm.h``.
"""
import concurrent.futures as cf
import hashlib
import os
import platform
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libspmm.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-O3",
          "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]
# Per-file flags (none at present).
PER_FILE = {}


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC)
                  if f.endswith((".cu", ".cpp")))


def _flags(src, extra):
    lang = ["-x", "cu"] if src.endswith(".cu") else ["-x", "c++"]
    return ARCH + COMMON + PER_FILE.get(os.path.basename(src), []) + list(extra) + lang


def _header_bytes():
    inc = os.path.join(ROOT, "include")
    paths = [os.path.join(d, f) for d in (CSRC, inc) for f in sorted(os.listdir(d))
             if f.endswith((".h", ".cuh"))]
    return b"".join(os.path.basename(p).encode() + open(p, "rb").read() for p in paths)


def _key(*parts):
    h = hashlib.sha256(platform.machine().encode())
    for p in parts:
        h.update(b"\0" + (p if isinstance(p, bytes) else p.encode()))
    return h.hexdigest()


def _fresh(path, key):
    """Whether ``path`` was built from what ``key`` stands for."""
    try:
        return os.path.exists(path) and open(path + ".key").read() == key
    except OSError:
        return False


def _run(cmd, out, key):
    """Runs a build command that writes to a name beside ``out``, then puts
    the result and its key in place."""
    tmp = out + ".tmp%d" % os.getpid()
    r = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
    if r.stderr.strip():
        sys.stderr.write(r.stderr)
    if os.path.exists(out + ".key"):
        os.remove(out + ".key")
    os.replace(tmp, out)
    with open(out + ".key", "w") as f:
        f.write(key)


def _compile(src, extra, headers, out_dir):
    obj = os.path.join(out_dir, os.path.basename(src) + ".o")
    key = _key(open(src, "rb").read(), headers, " ".join(_flags(src, extra)))
    if not _fresh(obj, key):
        _run([NVCC] + _flags(src, extra) + ["-c", src], obj, key)
    return obj, key


def build(verbose=False, extra=()):
    """Compiles what is not up to date and links the library.  An object is up
    to date by the content of its source, the headers and its flags: times say
    nothing of flags, and the record formats that two objects share have to
    come from one state of the headers.  Objects of other flags (``extra``) lie
    in a folder of their own."""
    extra = list(extra)
    out_dir = os.path.join(OUT_DIR, "flags-" + _key(" ".join(extra))[:12]) if extra else OUT_DIR
    os.makedirs(out_dir, exist_ok=True)
    srcs, headers = sources(), _header_bytes()
    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        built = list(ex.map(lambda s: _compile(s, extra, headers, out_dir), srcs))
    key = _key(*[k for _, k in built])
    if not _fresh(LIB, key):
        _run([NVCC] + ARCH + ["-shared"] + [o for o, _ in built], LIB, key)
        if verbose:
            print(LIB)
    return LIB


if __name__ == "__main__":
    extra = sys.argv[1:]
    print(build(verbose=True, extra=extra))
