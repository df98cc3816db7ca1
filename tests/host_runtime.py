"""Run a piece of host code against libmc.so with the CUDA runtime replaced by tests/cuda/fake_cudart.c, in a process of
its own (no GPU, no torch): what the library launches, in which order and with which attributes, and what
it does when a launch fails."""
import json
import os
import subprocess
import sys
import tempfile

from conftest import ROOT

PRELUDE = '''
import ctypes, json
from paper_0903_3053_gb300 import mc
fake = ctypes.CDLL(None)
fake.fake_log.restype = ctypes.c_char_p
lib = mc.load()
mc._load_van()
keep = []

def memory(nbytes):
    """256-byte aligned host memory that stands in for device memory."""
    buf = ctypes.create_string_buffer(int(nbytes) + 256)
    keep.append(buf)
    return ctypes.c_void_p((ctypes.addressof(buf) + 255) & ~255)

def stream():
    s = ctypes.c_void_p()
    assert fake.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0
    return s

def batch(chains, layout=0, cap=1024, st=None):
    arr = (mc.mc_chain_desc * len(chains))(*[c.desc() for c in chains])
    n = mc.mc_workspace_bytes(chains, layout, cap)
    ctx = ctypes.c_void_p()
    assert lib.mc_batch_init(ctypes.byref(ctx), len(chains), arr, layout, cap, memory(n), n, st) == 0
    return ctx

def group(ctxs, st=None):
    arr = (ctypes.c_void_p * len(ctxs))(*[c.value for c in ctxs])
    n = lib.mc_group_workspace_bytes(len(ctxs), arr)
    g = ctypes.c_void_p()
    assert lib.mc_group_create(ctypes.byref(g), len(ctxs), arr, memory(n), n, st) == 0
    return g

def van(L, n, depth, st=None):
    nb = lib.mc_van_workspace_bytes(L, n, depth)
    w = ctypes.c_void_p()
    return lib.mc_van_create(ctypes.byref(w), L, n, depth, 1, memory(nb), nb, st), w

def swept(ctx):
    v = ctypes.c_int64()
    assert lib.mc_get_sweep(ctx, ctypes.byref(v)) == 0
    return v.value

def launches():
    """What was launched since the last call: [name, blocks, threads, "programmatic" or "plain"], and ["graph"],
    ["end"], ["wait"]."""
    out = [l.split() for l in fake.fake_log().decode().splitlines()]
    fake.fake_clear()
    return out
'''


def run(script: str):
    """The value that `script` leaves in `result`."""
    with tempfile.TemporaryDirectory() as d:
        so = os.path.join(d, "fake_cudart.so")
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        subprocess.run([os.environ.get("CC", "gcc"), "-shared", "-fPIC", "-O1", "-I", os.path.join(cuda, "include"),
                        os.path.join(ROOT, "tests", "cuda", "fake_cudart.c"), "-o", so], check=True)
        from paper_0903_3053_gb300 import build
        if not build.up_to_date():
            build.build()
        r = subprocess.run([sys.executable, "-c", PRELUDE + script + "\nprint('RESULT ' + json.dumps(result))"], cwd=ROOT,
                           env=dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
        return json.loads(r.stdout.rsplit("RESULT ", 1)[1])
