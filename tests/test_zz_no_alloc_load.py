"""snerg_render_rays_noalloc loads every kernel it can launch at its first call on a device: a fresh
process makes one call without rays, and CUDA then reports each of the entry point's
kernels as loaded; a call of another block edge and of more than one wave of rays is captured,
and its replay gives what the plain call gives."""
import subprocess
import sys
import os

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes
import numpy as np
import torch
from paper_2103_14645_gb300 import renderer, synth

DEV = torch.device("cuda:0")
torch.zeros(1, device=DEV)
cu = ctypes.CDLL("libcuda.so.1")
lib = renderer.load_library()


class KernelNode(ctypes.Structure):         # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p),
                ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def ok(code):
    assert code == 0, code


def call(B, n, stream, rng):
    ind = np.arange(8, dtype=np.int32).reshape(2, 2, 2)
    atlas = rng.integers(0, 256, (8, B, B, B, 8), dtype=np.uint8)
    cams = synth.orbit_cameras(rng, [(400, 300)] * 2, 1.6, 50.0)
    desc = renderer.SceneDesc(2 * B, B, (ctypes.c_float * 3)(-1, -1, -1), 2.0, 40.0, (ctypes.c_float * 3)(1, 1, 1), 0, 0)
    t = [torch.from_numpy(a).to(DEV) for a in (ind, atlas, synth.random_pixels(rng, cams, n), synth.init_mlp(rng))]
    out = torch.full((n, 3), float("nan"), device=DEV)
    torch.cuda.synchronize()

    def launch(s):
        ok(lib.snerg_render_rays_noalloc(ctypes.byref(desc), t[0].data_ptr(), t[1].data_ptr(), 8, cams.ctypes.data, 2,
                                         t[2].data_ptr(), n, t[3].data_ptr(), out.data_ptr(), None, s))
    return launch, out


stream = torch.cuda.Stream()
s = ctypes.c_void_p(stream.cuda_stream)
first, _ = call(8, 0, s, np.random.default_rng(0))
first(s)
torch.cuda.synchronize()

# the entry point's module, from a kernel of a captured call without rays
graph = ctypes.c_void_p()
ok(cu.cuStreamBeginCapture_v2(s, 0))
first(s)
ok(cu.cuStreamEndCapture(s, ctypes.byref(graph)))
count = ctypes.c_size_t(0)
ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(count)))
nodes = (ctypes.c_void_p * count.value)()
ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)))
node = KernelNode()
ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[0]), ctypes.byref(node)))
func, module = ctypes.c_void_p(node.func), ctypes.c_void_p()
if not func:
    ok(cu.cuKernelGetFunction(ctypes.byref(func), ctypes.c_void_p(node.kern)))
ok(cu.cuFuncGetModule(ctypes.byref(module), func))
n_funcs = ctypes.c_uint(0)
ok(cu.cuModuleGetFunctionCount(ctypes.byref(n_funcs), module))
funcs = (ctypes.c_void_p * n_funcs.value)()
ok(cu.cuModuleEnumerateFunctions(funcs, n_funcs, module))
state = {}
for f in funcs:
    name, loaded = ctypes.c_char_p(), ctypes.c_int(-1)
    ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(f)))
    ok(cu.cuFuncIsLoaded(ctypes.byref(loaded), ctypes.c_void_p(f)))
    if b"noalloc" in name.value:
        state[name.value.decode()] = loaded.value
assert len(state) == 12, sorted(state)                # two of the maps, two for each of five block builds
late = [k for k, v in state.items() if v != 1]
assert not late, late

launch, out = call(32, 150000, s, np.random.default_rng(1))
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=stream):
    launch(s)
g.replay()
torch.cuda.synchronize()
got = out.clone()
out.fill_(float("nan"))
launch(s)
torch.cuda.synchronize()
assert bool(torch.isfinite(got).all()) and torch.equal(got, out)
print("loaded")
'''


def test_the_first_call_loads_every_kernel():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CUDA_MODULE_LOADING="LAZY"))
    assert r.returncode == 0 and r.stdout.strip().endswith("loaded"), r.stdout + r.stderr
