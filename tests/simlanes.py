"""ctr_simulate on the CPU: api.cu and sim.cu compiled as C++ on the fibers of
tests/host/lanes.h (launches become calls), so the simulator's kernels run
without a GPU, their lanes in any order and their memory accesses checked."""
import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from conftest import ROOT
from paper_2609_16206_gb300 import ctr

CSRC = os.path.join(ROOT, "paper_2609_16206_gb300", "csrc")
HOST = os.path.join(ROOT, "tests", "host")
_LAUNCH = re.compile(r"(\w+(?:<[^;<>]*>)?)<<<(.+?), ([^,;]+?), 0, stream>>>\((.*?)\);")
# launches of the other translation units: not called here
_STUBS = "\n".join(f"cudaError_t {f} {{ return cudaErrorNotSupported; }}" for f in (
    "launch_trace(const TraceParams&, cudaStream_t)", "launch_score(const ScoreParams&, cudaStream_t)",
    "launch_stream_probe(const ScoreParams&, cudaStream_t)", "launch_goodput(const GoodputParams&, cudaStream_t)")) + """
cudaError_t launch_mix_table(uint64_t* t, int64_t n, cudaStream_t)
{
    for (int64_t i = 0; i < 2 * n; ++i) t[i] = mix64((uint64_t(i < n ? 2 : 3) << 56) ^ (uint64_t)(i < n ? i : i - n));
    return cudaSuccess;
}"""


def build(out_dir):
    gxx = shutil.which("g++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    with open(os.path.join(CSRC, "sim.cu")) as f:
        sim, n = _LAUNCH.subn(r"lanes::launch(\2, \3, [&] { \1(\4); });", f.read())
    assert n == 6 and "<<<" not in sim, n
    with open(os.path.join(out_dir, "sim.cpp"), "w") as f:
        f.write('#include "lanes.h"\n#include "ctr_internal.cuh"\n#define asm(...) r = 1.0f / (float)d\n' + sim +
                "\n#undef asm\n#include \"api.cu\"\nnamespace ctr {\n" + _STUBS + "\n}\n")
    flags = ["-std=c++17", "-O1", "-DCTR_BOUNDS_CHECK=1", "-fPIC", "-w", "-I", HOST, "-I", CSRC, "-I", cuda]
    objs = []
    for src, extra in ((os.path.join(out_dir, "sim.cpp"), ["-fsanitize=thread"]), (os.path.join(HOST, "lanes.cpp"), [])):
        objs.append(os.path.join(out_dir, os.path.basename(src) + ".o"))
        subprocess.run([gxx, *flags, *extra, "-c", src, "-o", objs[-1]], check=True)
    so = os.path.join(out_dir, "libsimlanes.so")
    subprocess.run([gxx, "-shared", "-Wl,-Bsymbolic", "-o", so, *objs], check=True)
    L = C.CDLL(so)
    vp, i32, i64 = C.c_void_p, C.c_int32, C.c_int64
    L.ctr_workspace_bytes.argtypes = [i32, C.POINTER(ctr.CtrSimCfg), i64, i64]
    L.ctr_workspace_bytes.restype = C.c_size_t
    L.ctr_simulate.argtypes = [C.POINTER(ctr.CtrSimCfg), C.POINTER(ctr.CtrCostConsts), i32, C.POINTER(i32), i32,
                               ctr.CtrRequests, i32, i64, vp, vp, vp, vp, vp, vp, vp, vp, vp, C.c_size_t, vp]
    L.lanes_faults.restype = C.c_longlong
    return L


def simulate(L, sc, sets, pols, traces, order=0, ws_rows=None):
    """One call over host traces (a list of dicts of equal length): statuses, checksums, times and routes, the number of
    accesses that nothing orders and of blocks stuck at different collectives.  ws_rows: a workspace for that many rows in place of all."""
    n, R = len(traces[0]["arrival_us"]), len(traces)
    rows = R * len(sets) * len(pols)
    dts = {"arrival_us": np.int64, "prompt_len": np.int32, "true_out": np.int32, "pred_out": np.int32, "slo_class": np.uint8}
    tr = {k: np.ascontiguousarray(np.stack([t[k] for t in traces]), dtype=d) for k, d in dts.items()}
    res = {"t_first_us": np.full((rows, n), -7, np.int64), "t_done_us": np.full((rows, n), -7, np.int64),
           "i_pre": np.zeros((rows, n), np.uint8), "i_dec": np.zeros((rows, n), np.uint8),
           "status": np.full(rows, 99, np.int32), "hash": np.zeros(rows, np.uint64)}
    cfg = ctr.sim_cfg_struct(sc)
    nbytes = L.ctr_workspace_bytes(0, C.byref(cfg), ws_rows or rows, n)
    ws = np.zeros(nbytes + 256, np.uint8)
    at = ws.ctypes.data + (-ws.ctypes.data) % 256
    L.lanes_order(order)
    p = lambda a: a.ctypes.data
    rc = L.ctr_simulate(C.byref(cfg), ctr.consts_array(sets), len(sets), (C.c_int32 * len(pols))(*pols), len(pols),
                        ctr.CtrRequests(*(p(tr[k]) for k in dts)), R, n, p(res["i_pre"]), p(res["i_dec"]),
                        p(res["t_first_us"]), p(res["t_done_us"]), p(res["hash"]), p(res["status"]), None, None, at, nbytes,
                        None)
    stuck = C.c_longlong()
    races = L.lanes_faults(C.byref(stuck))
    assert rc == ctr.CTR_OK
    return res, races, stuck.value
