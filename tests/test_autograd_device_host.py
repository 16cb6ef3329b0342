"""The layers' kernels go to the device and stream of their tensors, not to the current device. On the CPU, in a child process: the
device functions that the module calls and the kernel's launcher are replaced by recorders (LD_PRELOAD), the tensors claim to be on
cuda:1 but lie in host memory, and the framework's own operators on them are Python functions."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKES = r"""
#include <stdint.h>
#include <stdio.h>
static int8_t current = 0;
struct Stream { int8_t type, index, pad[6]; int64_t id; };
int8_t _ZN3c104cuda14ExchangeDeviceEa(int8_t d) { int8_t old = current; if (d >= 0) current = d; return old; }
int8_t _ZN3c104cuda14MaybeSetDeviceEa(int8_t d) { return _ZN3c104cuda14ExchangeDeviceEa(d); }
int _ZN3c104cuda9GetDeviceEPa(int8_t* d) { *d = current; return 0; }
int _ZN3c104cuda9SetDeviceEab(int8_t d, _Bool force) { current = d; return 0; }
int8_t _ZN3c104cuda12device_countEv(void) { return 2; }
struct Stream _ZN3c104cuda20getCurrentCUDAStreamEa(int8_t d) { struct Stream s = {1, d < 0 ? current : d, {0}, 0}; return s; }
void* _ZNK3c104cuda10CUDAStream6streamEv(const struct Stream* s) { return (void*)(intptr_t)(100 + s->index); }
int _ZN4sdgp19launch_relu_maxpoolEPKvlllliPvP11CUstream_st(const void* x, int64_t b, int64_t h, int64_t w, int64_t k, int dtype, void* y,
                                                           void* stream) {
  printf("launch on device %d, stream of device %d\n", current, (int)((intptr_t)stream - 100));
  fflush(stdout);
  return 0;
}
int recorded_device(void) { return current; }
"""

CHILD = r"""
import ctypes
import torch
import torch.utils.dlpack

torch.cuda._lazy_init = lambda: None


class DLTensor(ctypes.Structure):
    _fields_ = [("data", ctypes.c_void_p), ("device_type", ctypes.c_int), ("device_id", ctypes.c_int), ("ndim", ctypes.c_int),
                ("code", ctypes.c_uint8), ("bits", ctypes.c_uint8), ("lanes", ctypes.c_uint16), ("shape", ctypes.c_void_p),
                ("strides", ctypes.c_void_p), ("offset", ctypes.c_uint64)]


class Managed(ctypes.Structure):
    _fields_ = [("t", DLTensor), ("ctx", ctypes.c_void_p), ("deleter", ctypes.c_void_p)]


ctypes.pythonapi.PyCapsule_New.restype = ctypes.py_object
ctypes.pythonapi.PyCapsule_New.argtypes = [ctypes.c_void_p, ctypes.c_char_p, ctypes.c_void_p]
kept = []


def on_cuda1(host):
    shape = (ctypes.c_int64 * host.dim())(*host.shape)
    strides = (ctypes.c_int64 * host.dim())(*host.stride())
    m = Managed(DLTensor(host.data_ptr(), 2, 1, host.dim(), 4, 16, 1, ctypes.addressof(shape), ctypes.addressof(strides), 0), None, None)
    kept.extend((host, shape, strides, m))
    return torch.utils.dlpack.from_dlpack(ctypes.pythonapi.PyCapsule_New(ctypes.addressof(m), b"dltensor", None))


def channels_last(*shape):
    return on_cuda1(torch.zeros(shape, dtype=torch.bfloat16).contiguous(memory_format=torch.channels_last))


ops = torch.library.Library("aten", "IMPL")
ops.impl("convolution", lambda x, w, *rest: channels_last(2, 64, 8, 8), "CUDA")
ops.impl("empty.memory_format", lambda size, **kw: channels_last(*size), "CUDA")
from paper_2202_00774_b200 import autograd

y = autograd.sdgp_conv2d_relu(channels_last(2, 64, 8, 8), channels_last(64, 64, 3, 3), 1, 1, pool=True)
print(tuple(y.shape), y.device, "current device", ctypes.CDLL(None).recorded_device(), flush=True)
import os
os._exit(0)  # (no tear-down of the pretended device)
"""


def test_pooled_layer_launches_on_the_device_of_its_tensors(tmp_path):
    source, fakes = tmp_path / "fakes.c", tmp_path / "fakes.so"
    source.write_text(FAKES)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", "-o", str(fakes), str(source)])
    env = dict(os.environ, LD_PRELOAD=str(fakes), PYTHONPATH=ROOT)
    done = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
    assert done.stdout.splitlines() == ["launch on device 1, stream of device 1", "(2, 64, 4, 4) cuda:1 current device 0"]
