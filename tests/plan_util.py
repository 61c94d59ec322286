"""The launch planner (csrc/agx_plan.cu) on the CPU: built with g++ behind a function that prints a plan."""
from __future__ import annotations

import ctypes
import functools
import os
import subprocess
import tempfile
from dataclasses import dataclass
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parent.parent
KINDS = ("small1", "small2", "small4", "stream", "tile", "simt")

_WRAPPER = r'''
#include <stdio.h>
#include "agx_plan.cu"
// clusters of 2 .. 16 CTAs that a B200 holds, one CTA per SM (8-page stages, 64-row blocks) and two (4-page stages)
static int clusters(int mt, int kw, int n) {
    static const int one[] = {74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7}, two[] = {148, 93, 71, 56, 45, 37, 33, 30, 26, 21, 21, 17, 14, 14, 14};
    return n < 2 || n > 16 ? 0 : (kw == 4 && mt < 4 ? two : one)[n - 2];
}
extern "C" int accept_chunks(int sms, int rows, int vocab, int elem_bytes, int aligned) { return agx::accept_chunks(sms, rows, vocab, elem_bytes, aligned != 0); }
extern "C" int plan(int hq, int hkv, int d, int dtype, int sms, int B, const int* P, const int* Q, int stride, char* out, int out_bytes) {
    const agx_config cfg = {hq, hkv, d, 16, dtype, 0.f};
    agx::Plan pl;
    char err[512] = "";
    const agx_status st = agx::build_plan(agx::plan_config(cfg, sms, clusters), B, P, Q, stride, pl, err, sizeof err);
    int n = snprintf(out, out_bytes, "%d %lld %s\n", st, pl.part_entries, err);
    for (const agx::Launch& l : pl.launches) {
        n += snprintf(out + n, out_bytes - n, "%d %d %d %d %d %d", (int)l.kind, l.kw, l.cluster, (int)l.lean_merge, l.num_items, l.total_rows);
        for (const agx::SeqPlan& s : l.seqs)
            n += snprintf(out + n, out_bytes - n, " %d %d %d %d %d %d", s.seq_index, s.nsplit, s.split_tokens, s.row_chunks, s.item0, s.part_base);
        n += snprintf(out + n, out_bytes - n, "\n");
    }
    return n;
}
'''


@dataclass
class Seq:
    index: int
    nsplit: int
    split_tokens: int
    row_chunks: int
    item0: int
    part_base: int


@dataclass
class Launch:
    kind: str
    kw: int
    cluster: int
    lean: bool
    items: int
    rows: int
    seqs: list


@dataclass
class Plan:
    status: int
    part_entries: int
    error: str
    launches: list

    def kind_of(self, seq: int) -> str:
        return next(l.kind for l in self.launches for s in l.seqs if s.index == seq)


@functools.cache
def _lib():
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    with tempfile.TemporaryDirectory() as tmp:
        src, out = Path(tmp) / "plan.cpp", Path(tmp) / "plan.so"
        src.write_text(_WRAPPER)
        subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-shared", "-fPIC", "-w", f"-I{cuda}", f"-I{ROOT / 'include'}",
                        f"-I{ROOT / 'paper_2605_10380_b200' / 'csrc'}", str(src), "-o", str(out)], check=True)
        return ctypes.CDLL(str(out))


def plan(P, Q, hq=32, hkv=8, d=128, dtype="bf16", sms=148, stride=-1) -> Plan:
    P, Q = np.asarray(P, np.int32), np.asarray(Q, np.int32)
    buf = ctypes.create_string_buffer(512 * len(P) + 4096)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    _lib().plan(hq, hkv, d, 0 if dtype == "bf16" else 1, sms, len(P), ptr(P), ptr(Q), stride, buf, len(buf))
    head, *lines = buf.value.decode().split("\n")
    status, entries, error = head.split(" ", 2)
    launches = []
    for line in filter(None, lines):
        v = [int(x) for x in line.split()]
        launches.append(Launch(KINDS[v[0]], v[1], v[2], bool(v[3]), v[4], v[5], [Seq(*v[i:i + 6]) for i in range(6, len(v), 6)]))
    return Plan(int(status), int(entries), error, launches)


def accept_chunks(rows, vocab, elem_bytes=2, aligned=True, sms=148) -> int:
    return _lib().accept_chunks(sms, rows, vocab, elem_bytes, int(aligned))
