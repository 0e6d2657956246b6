"""The native side of the hot calls: what it cannot take an address of is a Python error, never the end of the
process, and subclasses and torch function modes are asked as they are through Python."""
import functools
import os
import subprocess
import sys

import pytest

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
