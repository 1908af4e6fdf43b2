"""Host memory that runs out inside an entry point: a status, no exception across the C boundary."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# operator new that throws while `failing` is set
PRELOAD = r"""
#include <cstdlib>
#include <new>
extern "C" { int failing = 0; }
void* operator new(std::size_t n) {
  void* p = failing ? nullptr : std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CALLS = r"""
import ctypes, sys
import torch
from paper_2403_03507_b200 import binding as gb
failing = ctypes.c_int.in_dll(ctypes.CDLL(sys.argv[1]), "failing")
layers = [gb.Layer(gb.make_config(64, 96, 8, w_dtype="f32", g_dtype="f32", auto_refresh=False)) for _ in range(2)]
Ws, Gs = [torch.randn(64, 96, device="cuda") for _ in range(2)], [torch.randn(64, 96, device="cuda") for _ in range(2)]
for l in layers:
    l.set_projector(torch.linalg.qr(torch.randn(64, 8, device="cuda"))[0])
batch = gb.Batch(layers, Ws, Gs)
host = gb.HostBatch(layers, [w.cpu().pin_memory() for w in Ws], [g.cpu().pin_memory() for g in Gs])
calls = {"batch": lambda: batch.galore_step_batch(1e-2), "host": lambda: host.galore_step_host_batch(1e-2),
         "refresh": lambda: layers[0].galore_refresh_projector(Gs[0])}
for name, call in calls.items():
    call()
    torch.cuda.synchronize()
    failing.value = 1
    try:
        call()
        status = 0
    except gb.GaloreError as e:
        status = e.status
    finally:
        failing.value = 0
    assert status == gb.ERR_INVALID_ARG, (name, status)
    call()
    torch.cuda.synchronize()
print("statuses as stated")
"""


def test_entry_points_return_a_status_when_host_memory_runs_out(tmp_path):
    src, so = tmp_path / "fail.cpp", tmp_path / "libfail.so"
    src.write_text(PRELOAD)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-o", str(so), str(src)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CALLS, str(so)], capture_output=True, text=True, env=env, cwd=ROOT, timeout=300)
    assert r.returncode == 0 and "statuses as stated" in r.stdout, r.stdout + r.stderr
