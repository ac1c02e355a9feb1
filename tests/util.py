"""Shared helpers of the tests: marshal a synthetic workload into oracle inputs."""
from __future__ import annotations

import numpy as np

from paper_2604_26209_b200 import synth
from oracle import capi


def widen(t):
    """bf16-bit tensors -> fp32 arrays (exact)."""
    return {k: synth.bf16_bits_to_f32(v) for k, v in t.items()}


def oracle_step(s, t_bits, n_threads=0, rows=None):
    """Run the oracle on structure ``s`` with bf16-bit tensors ``t_bits`` (per-slot q/k_new/v_new)."""
    g = s.geom
    meta = capi.build_meta(s.doc_prefix_len, s.doc_branch_cnt, s.slot_depth, s.slot_alive, g.suffix_cap, s.pos_gap)
    f = widen(t_bits)
    act = meta.active_slot[: meta.n_active]
    out = capi.decode_step(g, meta, s.doc_prefix_len, f["q"][act], f["k_new"][act], f["v_new"][act],
                           f["prefix_k"], f["prefix_v"], f["suffix_k"], f["suffix_v"],
                           n_threads=n_threads, rows=rows)
    return meta, out


def err_stats(got, want):
    d = np.abs(np.asarray(got, dtype=np.float64) - np.asarray(want, dtype=np.float64))
    return (float(d.max()) if d.size else 0.0, float(d.mean()) if d.size else 0.0)


def copy_warps_rule(build_dir):
    """The host rule that picks a decode launch's kernel, compiled from its header: f(n_docs, max_rows, total_prefix, G, Hkv, D, n_sm, work_cap,
    part_cap, new_tokens = 1) -> (copy warps, expected units)."""
    import ctypes
    import os
    import subprocess
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, lib = os.path.join(build_dir, "rule.cpp"), os.path.join(build_dir, "rule.so")
    with open(src, "w") as f:
        f.write('#include "copy_warps.h"\nextern "C" long long rule(const hpd::StepSize* s, int* pay)\n'
                "{ *pay = hpd::copy_warps_pay(*s); return hpd::average_unit(*s).units; }\n")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", os.path.join(root, "paper_2604_26209_b200", "csrc"), src,
                    "-o", lib], check=True)
    fn = ctypes.CDLL(lib).rule
    fn.restype = ctypes.c_longlong

    def call(*sizes, new_tokens=1):
        pay = ctypes.c_int()
        units = fn((ctypes.c_int * 10)(*sizes, new_tokens), ctypes.byref(pay))
        return bool(pay.value), units
    return call
