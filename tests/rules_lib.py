"""The library's host rules (csrc/rules.h, plain C++) compiled for the tests."""
import ctypes
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "rules.h"
using namespace nlos;
extern "C" {
int rows_per_bin(double s) { return moment_rows_per_bin(s); }
int fits(double s) { return moments_fit(s); }
int max_j() { return kMomMaxJ; }
int max_taps() { return kMomTaps; }
int forward_mom(double s, uint64_t P, uint32_t B) { return forward_moments(s, P, B); }
uint32_t pairs_of_block(uint32_t most, uint32_t t, uint32_t w, uint32_t n, uint32_t sms) {
  return block_pairs(most, t, w, n, sms);
}
uint64_t pass_runs(uint64_t runs, uint64_t n_blk) { return list_pass_runs(runs, n_blk); }
uint64_t list_entries() { return kListEntries; }
int adjoint_mom(double s, uint64_t P, uint32_t B) { return adjoint_moments(s, P, B); }
}
"""


def load():
    d = tempfile.mkdtemp()
    src, so = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
    with open(src, "w") as f:
        f.write(SRC)
    inc = os.path.join(ROOT, "paper_2506_03747_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + inc, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.rows_per_bin.argtypes = lib.fits.argtypes = [ctypes.c_double]
    lib.forward_mom.argtypes = lib.adjoint_mom.argtypes = [ctypes.c_double, ctypes.c_uint64, ctypes.c_uint32]
    lib.pass_runs.argtypes = [ctypes.c_uint64, ctypes.c_uint64]
    lib.pass_runs.restype = lib.list_entries.restype = ctypes.c_uint64
    return lib
