"""The native side of the hot calls: what it cannot take an address of is a Python error, never the end of the
process, and subclasses and torch function modes are asked as they are through Python."""
import functools
import os
import subprocess
import sys

import pytest

from paper_2209_07663_b200 import binding as mb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Every case runs in a process of its own, forked after the imports, because what is tested for is that it lives on.
# The table is a null handle, which the library refuses (MonoError) when a call gets that far.
PROGRAM = """
import os, sys, warnings
import torch
from torch.fx.experimental.proxy_tensor import make_fx
from paper_2209_07663_b200 import binding as mb
warnings.simplefilter("ignore")
mb.load_library()
ids, off, x = torch.zeros(4, dtype=torch.int64), torch.tensor([0, 4]), torch.zeros(4)
seen = []

class Listening(torch.overrides.TorchFunctionMode):
    def __torch_function__(self, f, types, args=(), kwargs=None):
        seen.append(f.__name__)
        return f(*args, **(kwargs or {}))

class Answering(torch.Tensor):
    def data_ptr(self):
        raise KeyError("asked")

def push(g):
    mb.mono_apply_grads(0, ids, 4, off, 1, g, 0)
    return g.sum()

def pull(g):
    mb.mono_lookup_pool(0, ids, 4, off, 1, g)
    return g.sum()

def grouped(g):
    mb.mono_group_lookup_pool([0], [ids], [off], [g])
    return g.sum()

def listened():
    with Listening():
        try:
            push(x)
        except mb.MonoError:
            pass
    raise LookupError(seen.count("data_ptr"))

CASES = {}
for name, f in (("push", push), ("pull", pull), ("grouped", grouped)):
    CASES.update({
        name + " vmap": lambda f=f: torch.vmap(f)(torch.zeros(2, 4)),
        name + " grad": lambda f=f: torch.func.grad(f)(x),
        name + " jvp": lambda f=f: torch.func.jvp(f, (x,), (x,)),
        name + " csr": lambda f=f: f(torch.eye(4).to_sparse_csr()),
        name + " mkldnn": lambda f=f: f(x.to_mkldnn()),
        name + " fake": lambda f=f: make_fx(f, tracing_mode="fake")(x),
        name + " strided": lambda f=f: f(torch.zeros(4, 4).t()),
        name + " subclass": lambda f=f: f(x.as_subclass(Answering)),
        name + " plain": lambda f=f: f(x),
    })
CASES["listened"] = listened
for name, case in CASES.items():
    sys.stdout.flush()
    child = os.fork()
    if child == 0:
        try:
            case()
            print(name + ": returned", flush=True)
        except Exception as e:
            print(name + ": " + type(e).__name__, e if isinstance(e, LookupError) else "", flush=True)
        os._exit(0)
    status = os.waitpid(child, 0)[1]
    if status:
        print(name + ": ended with status", status, flush=True)
"""


@functools.lru_cache(maxsize=1)
def outcomes():
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PYTHONPATH=ROOT, CUDA_VISIBLE_DEVICES=""), cwd=ROOT)
    assert r.returncode == 0, r.stderr
    return dict(line.split(": ", 1) for line in r.stdout.strip().splitlines())


@pytest.mark.parametrize("call", ["push", "pull", "grouped"])
@pytest.mark.parametrize("what,want", [
    ("vmap", "RuntimeError"), ("grad", "RuntimeError"), ("jvp", "RuntimeError"), ("csr", "RuntimeError"),
    ("mkldnn", "RuntimeError"), ("fake", "RuntimeError"), ("strided", "ValueError"), ("subclass", "KeyError 'asked'"),
    ("plain", "MonoError"),
])
def test_what_has_no_address_is_a_python_error(call, what, want):
    assert outcomes()[f"{call} {what}"].strip() == want


def test_a_torch_function_mode_hears_of_the_tensors():
    assert outcomes()["listened"] == "LookupError 3"


# 2^23 tables (a block of zeros stands for each: nothing is read of it but its device) and room for half of the first
# host vector that describes them.
STARVED = """
import ctypes, resource
from paper_2209_07663_b200 import binding as mb
lib = mb.load_library()
n = 1 << 23
mb.mono_group_prepare_push([], [], [])
zeros = ctypes.create_string_buffer(1 << 16)
tables = (ctypes.c_void_p * n)(*([ctypes.addressof(zeros)] * n))
handles = [0] * n
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + 4 * n, resource.getrlimit(resource.RLIMIT_AS)[1]))
empty = ctypes.c_void_p()
print(lib.mono_group_prepare_push(n, tables, empty, empty, empty, empty, empty))
print(lib.mono_group_lookup_pool(n, tables, empty, empty, empty, empty, empty, empty))
print(lib.mono_group_apply_grads(n, tables, empty, empty, empty, empty, empty, 0, empty))
try:
    mb.mono_group_prepare_push(handles, handles, handles)
except MemoryError:
    print("MemoryError")
"""


def test_a_grouped_call_without_host_memory_is_an_error():
    r = subprocess.run([sys.executable, "-c", STARVED], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PYTHONPATH=ROOT, CUDA_VISIBLE_DEVICES=""), cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == [str(mb.MONO_ERR_NOMEM)] * 3 + ["MemoryError"]


# What a caller with arrays and addresses needs is the library alone.
WITHOUT_TORCH = """
import os, sys
if sys.argv[1] == "absent":
    sys.modules["torch"] = None                     # import torch raises
import numpy as np
from paper_2209_07663_b200 import binding as mb
mb.load_library()
ids, off, out = np.zeros(4, np.uint64), np.array([0, 4]), np.zeros(4, np.float32)
calls = [lambda: mb.mono_lookup_pool_host(0, ids, 4, off, 1, out), lambda: mb.mono_apply_grads_host(0, ids, 4, off, 1, out, 0),
         lambda: mb.mono_lookup_pool(0, 4096, 4, 4096, 1, 4096), lambda: mb.mono_lookup_pool_noalloc(0, ids, 4, off, 1, out),
         lambda: mb.mono_apply_grads(0, ids, 4, off, 1, out, 0), lambda: mb.mono_prepare_push(0, ids, 4, off, 1),
         lambda: mb.mono_group_ahead(0, ids, 4, off, 1), lambda: mb.mono_expire(0, 1), lambda: mb.mono_expire_slice(0, 1, 0, 4),
         lambda: mb.mono_fence(0), lambda: mb.mono_apply_grads(0, ids[::2], 2, off, 1, out, 0)]
def all_of_them():
    for call in calls:
        try:
            call()
        except Exception as e:
            print(type(e).__name__)
all_of_them()
mb.mono_group_prepare_push([], [], [])
mb.mono_group_lookup_pool([], [], [], [])
mb.mono_group_apply_grads([], [], [], [], 0)
print(sys.modules.get("torch") is None, mb._native is None)
if sys.argv[1] == "later":
    import torch
    all_of_them()
    print(sys.modules.get("torch") is None, mb._native is None)
"""


@pytest.mark.parametrize("torch_is", ["absent", "later"])
def test_arrays_need_neither_torch_nor_the_extension(torch_is):
    r = subprocess.run([sys.executable, "-c", WITHOUT_TORCH, torch_is], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PYTHONPATH=ROOT, CUDA_VISIBLE_DEVICES=""), cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    each = ["MonoError"] * 10 + ["ValueError"]
    assert r.stdout.split() == each + ["True", "True"] + (each + ["False", "False"] if torch_is == "later" else [])


def test_another_torch_gets_an_extension_of_its_own(monkeypatch):
    from paper_2209_07663_b200 import build
    import torch
    mine, made = build.build_native(), []

    def compiler(cmd):
        made.append(cmd[cmd.index("-o") + 1])
        open(made[-1], "w").close()
    monkeypatch.setattr(build.subprocess, "check_call", compiler)
    assert build.build_native() == mine and not made           # up to date
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    theirs = build.build_native()
    os.unlink(theirs)
    assert made and theirs != mine
    with pytest.raises(RuntimeError, match="missing"):
        mb._load_native(mb.load_library())
