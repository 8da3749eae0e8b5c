"""ctr_simulate and ctr_goodput on the CPU: api.cu, sim.cu and goodput.cu compiled
as C++ on the fibers of tests/host/lanes.h (launches become calls), so their
kernels run without a GPU, their lanes in any order and their memory accesses
checked."""
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
_LAUNCH = re.compile(r"(\w+(?:<[^;<>]*>)?)<<<(.+?), ([^,;]+?), ([^,;]+?), stream>>>\((.*?)\);")
# launches of the other translation units: not called here
_STUBS = "\n".join(f"cudaError_t {f} {{ return cudaErrorNotSupported; }}" for f in (
    "launch_trace(const TraceParams&, cudaStream_t)", "launch_score(const ScoreParams&, cudaStream_t)",
    "launch_stream_probe(const ScoreParams&, cudaStream_t)"))


def _source(name, launches):
    with open(os.path.join(CSRC, name)) as f:
        text, n = _LAUNCH.subn(r"lanes::launch(\2, \3, \4, [&] { \1(\5); });", f.read())
    assert n == launches and "<<<" not in text, (name, n)
    return re.sub(r"extern __shared__ (\w+) (\w+)\[\];", r"\1* const \2 = static_cast<\1*>(lanes::dynamic_shared());", text)


def build(out_dir):
    gxx = shutil.which("g++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    with open(os.path.join(out_dir, "kernels.cpp"), "w") as f:
        f.write('#include "lanes.h"\n#include "ctr_internal.cuh"\n#define asm(...) r = 1.0f / (float)d\n' +
                _source("sim.cu", 6) + "\n#undef asm\n#undef CTR_CK_FLAG_PARAM\n#undef CTR_CK_FLAG_ARG\n" +
                _source("goodput.cu", 2) + '\n#include "api.cu"\nnamespace ctr {\n' + _STUBS + "\n}\n")
    flags = ["-std=c++17", "-O1", "-DCTR_BOUNDS_CHECK=1", "-fPIC", "-w", "-I", HOST, "-I", CSRC, "-I", cuda]
    objs = []
    for src, extra in ((os.path.join(out_dir, "kernels.cpp"), ["-fsanitize=thread"]), (os.path.join(HOST, "lanes.cpp"), [])):
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
    L.ctr_goodput.argtypes = [C.POINTER(ctr.CtrSimCfg), ctr.CtrRequests, i32, i32, i64, vp, vp, vp, vp, vp, vp]
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


def goodput(L, sc, tr, t_first, t_done, order=0):
    """One call with the P99 TPOT, a row a replica: met, P99 TTFT and P99 TPOT per row, then as of simulate."""
    R, n = t_first.shape
    dts = {"arrival_us": np.int64, "prompt_len": np.int32, "true_out": np.int32, "pred_out": np.int32, "slo_class": np.uint8}
    tr = {k: np.ascontiguousarray(tr[k], dtype=d) for k, d in dts.items()}
    tf, td = (np.ascontiguousarray(x, dtype=np.int64) for x in (t_first, t_done))
    out = np.full((3, R), -9, np.int64)
    cfg = ctr.sim_cfg_struct(sc)
    L.lanes_order(order)
    rc = L.ctr_goodput(C.byref(cfg), ctr.CtrRequests(*(tr[k].ctypes.data for k in dts)), R, 1, n, tf.ctypes.data,
                       td.ctypes.data, *(out[i].ctypes.data for i in range(3)), None)
    stuck = C.c_longlong()
    races = L.lanes_faults(C.byref(stuck))
    assert rc == ctr.CTR_OK
    return out, races, stuck.value
