"""Set-up of kernels on several devices of one process, on the CPU against a
fake of the CUDA calls that it makes (no GPU)."""
import os
import subprocess
import sys

from paper_2609_14144_gb300 import _lib

# Two devices of compute capability 10.x; counts cudaFuncSetAttribute per device.
FAKE = r"""
static int device, calls[2];
void fake_set(int d) { device = d; }
int fake_calls(int d) { return calls[d]; }
static int encode(void) { return 0; }
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { (void)attr; (void)d; *v = 10; return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int v) { (void)f; (void)attr; (void)v; ++calls[device]; return 0; }
int cudaGetDriverEntryPointByVersion(const char* s, void** f, unsigned v, unsigned long long k, int* q) {
    (void)s; (void)v; (void)k; *f = (void*)encode; *q = 0; return 0;
}
int cudaGetLastError(void) { return 0; }
"""


def test_tcgen05_kernels_are_set_up_on_every_device(tmp_path):
    """A kernel's shared-memory limit belongs to a device: the engine created on
    the second device of a process sets it there too."""
    _lib.load(allow_build=True)
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)])
    code = f"""
import ctypes
fake, lib = ctypes.CDLL({str(so)!r}), ctypes.CDLL({_lib.lib_path()!r})
configure = lib._ZN2ee14configure_ummaEv
configure.restype = ctypes.c_bool
for d in (0, 1, 0, 1):
    fake.fake_set(d)
    assert configure()
print(fake.fake_calls(0), fake.fake_calls(1))
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=60,
                       env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr
    on = [int(x) for x in r.stdout.split()]
    assert on == [10, 10]  # three products and the attention at two head sizes, twice
