"""No entry point throws or ends the process when the host runs out of memory or threads (CPU; each case in a child process whose
address space is limited to what it already uses)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "paper_2602_05367_b200", "librabit.so")

PRELUDE = """
import ctypes, resource, sys
lib = ctypes.CDLL(sys.argv[1])
def limit_address_space():
    pages = int(open("/proc/self/statm").read().split()[0])
    resource.setrlimit(resource.RLIMIT_AS, (pages * resource.getpagesize() + (256 << 10), resource.RLIM_INFINITY))
"""

PLANS = """
out = (ctypes.c_int * 4000)()
head = (ctypes.c_int * 8)()
M, N = ctypes.c_int(0), ctypes.c_int(4096)
seen = []
def f16(i): return lib.rabit_selftest_f16_plan(2, 128 * (i + 1), 4096, 8, 148, out, 400)
def gemm(i):
    M.value = 128 * (i % 60 + 1)
    return lib.rabit_selftest_gemm_plan(1, ctypes.byref(M), ctypes.byref(N), 2, 0, 16 * (i // 60 + 1), 148, -1, head, out, 400)
call = {"f16": f16, "gemm": gemm}[sys.argv[2]]
call(0)
limit_address_space()
worst = 0
for i in range(250):
    worst = min(worst, call(i))
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
assert worst in (0, -1), worst
assert call(0) > 0
"""

PACK = """
M, N = 8192, 2048                       # 64 x 64 tiles: packed by several threads
lib.rabit_packed_bytes.restype = ctypes.c_size_t
size = lib.rabit_packed_bytes(1, M, N)
planes = (ctypes.c_uint32 * (M * N // 32))()
for i in range(0, len(planes), 7): planes[i] = (i * 2654435761) & 0xFFFFFFFF
g, h, image, again = (ctypes.c_uint16 * M)(), (ctypes.c_uint16 * N)(), (ctypes.c_char * size)(), (ctypes.c_char * size)()
lib.rabit_pack_host.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 3 + [ctypes.c_void_p, ctypes.c_size_t]
ctypes.memset(image, 1, size); ctypes.memset(again, 1, size)
limit_address_space()
rc = lib.rabit_pack_host(planes, g, h, 1, M, N, image, size)
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
assert rc == 0, rc                      # no thread to be had: the calling one does the work
assert lib.rabit_pack_host(planes, g, h, 1, M, N, again, size) == 0
assert image.raw == again.raw
"""


@pytest.mark.parametrize("body,args", [(PLANS, ["f16"]), (PLANS, ["gemm"]), (PACK, [])], ids=["f16 plans", "gemm plans", "packing"])
def test_entry_points_survive_without_host_memory(body, args):
    proc = subprocess.run([sys.executable, "-c", PRELUDE + body, LIB] + args, capture_output=True, text=True, timeout=120)
    assert proc.returncode == 0, (proc.returncode, proc.stderr[-1500:])
