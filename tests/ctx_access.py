"""A small shared library that reaches into a context (sta_internal.cuh's sta_ctx), for tests of what
the C-ABI does not show.  Built on first use, into a directory of the caller's."""
import ctypes as C
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parent.parent

SRC = r"""
#include "sta_internal.cuh"

extern "C" {
// a context without device state, for calls that end before any device work
void *ctx_new(void) {
    sta_ctx *x = new sta_ctx();
    x->c.h_fault = new unsigned int(0u);
    return x;
}
void ctx_delete(void *p) {
    sta_ctx *x = static_cast<sta_ctx *>(p);
    delete x->c.h_fault;
    delete x;
}
// the word that a rebuild whose wait ran out sets
void ctx_set_fault(void *p, unsigned int v) {
    *reinterpret_cast<volatile unsigned int *>(static_cast<sta_ctx *>(p)->c.h_fault) = v;
}
// lanes per node of the solve's plan (0: no plan yet)
int ctx_plan_lanes(void *p) {
    const sta::Ctx &c = static_cast<sta_ctx *>(p)->c;
    return c.cg ? c.cg_S : 0;
}
// polls of a solve's grid-wide waits at most
void ctx_set_spins(void *p, unsigned int n) { static_cast<sta_ctx *>(p)->c.cg_spins = n; }
unsigned int ctx_fault(void *p) {
    return *reinterpret_cast<volatile unsigned int *>(static_cast<sta_ctx *>(p)->c.h_fault);
}
}
"""


def load(directory):
    from paper_2605_11673_gb300 import build
    src, lib = Path(directory) / "ctx_access.cu", Path(directory) / "libctx_access.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-std=c++17", f"-I{ROOT / 'include'}",
                    f"-I{build.CSRC}", str(src), "-o", str(lib)], check=True, capture_output=True)
    L = C.CDLL(str(lib))
    L.ctx_new.restype = C.c_void_p
    L.ctx_delete.argtypes = [C.c_void_p]
    L.ctx_set_fault.argtypes = [C.c_void_p, C.c_uint]
    L.ctx_plan_lanes.argtypes = [C.c_void_p]
    L.ctx_set_spins.argtypes = [C.c_void_p, C.c_uint]
    L.ctx_fault.argtypes = [C.c_void_p]
    L.ctx_fault.restype = C.c_uint
    return L
