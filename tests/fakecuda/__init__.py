"""The library's host side on a fake CUDA runtime (fake_cudart.cpp), for tests
without a GPU: `run(code)` executes code in a child process that has loaded that
build, with `tsx` (the package), `np`, `lp(m, n)` (an LP), `solve(m, n, **options)`
(its status and statistics) and `fake` (the runtime's controls; `log()` gives the
launches so far as (device, kernel, blocks, threads, shared memory))."""
import hashlib
import os
import subprocess
import sys
import textwrap

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(os.path.dirname(HERE))

PRELUDE = """
import ctypes, re, sys
sys.path.insert(0, {root!r})
import numpy as np
from paper_2211_10979_gb300 import abi
fake = abi.load({lib!r})
import paper_2211_10979_gb300 as tsx
fake.fake_log.restype = ctypes.c_char_p
fake.fake_live.restype = fake.fake_peak.restype = ctypes.c_longlong

def log():
    out = []
    for line in fake.fake_log().decode().splitlines():
        *note, device, name, blocks, threads, smem = line.split()
        name = re.search(r"k_[a-z0-9_]*[a-z0-9]", re.sub(r"I?Li[0-9]+.*|I[df]E.*", "", name)).group()
        out.append((" ".join(note + [name]), int(device), int(blocks), int(threads), int(smem)))
    return out

def kernels():
    return [x[0] for x in log()]

def lp(m, n):
    return np.ones((m, n)), np.ones(m), np.ones(n)

def solve(m, n, device=0, **options):
    fake.fake_set_device(device)
    with tsx.Problem(*lp(m, n)) as pr:
        st = pr.solve(tsx.options(**options))
        return st, pr.stats()
"""


def build() -> str:
    """The library's sources without machine code for the device, linked with the
    fake runtime; rebuilt when a source changes."""
    sys.path.insert(0, ROOT)
    from paper_2211_10979_gb300 import build as b
    own = [os.path.join(HERE, f) for f in ("fake_cudart.cpp", "fake_kernels.cu")]
    digest = hashlib.sha256(b.source_digest().encode())
    for path in own:
        with open(path, "rb") as fh:
            digest.update(fh.read())
    digest = digest.hexdigest()[:16]
    objdir = os.path.join(b.PKG, "_build")
    out = os.path.join(objdir, f"libtabsimplex_fake_{digest}.so")
    if os.path.exists(out):
        return out
    os.makedirs(objdir, exist_ok=True)
    flags = ["-gencode", "arch=compute_103a,code=compute_103a", "-O1", "-std=c++17", "--fmad=false", "-Xcompiler",
             "-fPIC", "-I", b.INCLUDE, "-I", b.CSRC]
    jobs, objs = [], []
    for path in [os.path.join(b.CSRC, s) for s in b.SOURCES] + own:
        obj = os.path.join(objdir, f"fake_{os.path.basename(path)}.{os.getpid()}.o")
        jobs.append(subprocess.Popen([b.nvcc(), *flags, "-c", "-o", obj, path]))
        objs.append(obj)
    try:
        if any([j.wait() for j in jobs]):
            raise RuntimeError("the fake build does not compile")
        tmp = f"{out}.{os.getpid()}"
        subprocess.run([b.nvcc(), "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", tmp, *objs], check=True)
        os.replace(tmp, out)
    finally:
        for obj in objs:
            if os.path.exists(obj):
                os.remove(obj)
    return out


def run(code: str, timeout: float = 120.0) -> str:
    text = PRELUDE.format(root=ROOT, lib=build()) + textwrap.dedent(code)
    r = subprocess.run([sys.executable, "-c", text], capture_output=True, text=True, timeout=timeout)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    return r.stdout
