"""The step adjoint's work buffers when an allocation fails: the call reports it, and
so does the next one for as long as a buffer is missing (its kernels would read a
null pointer).  adj_alloc's own source, compiled for the host against a cudaMalloc
that fails on its n-th call."""
import ctypes
import os
import re
import subprocess

import pytest

import paper_2004_13887_gb300 as sph

CSRC = os.path.join(os.path.dirname(sph.__file__), "csrc")

HARNESS = r"""
#include <stddef.h>
#include <stdlib.h>
enum { cudaSuccess = 0, SPH_OK = 0, SPH_ERR_NOMEM = -5 };
namespace f64 { constexpr int ADJ_PLANES = 8; }
struct sph_ctx { size_t nf[5]; long N; int adjK; size_t fset, foff[5]; double *adjS, *adjW, *adjC; };
static int calls, fail_at;
static int cudaMalloc(void** p, size_t n) { if (++calls == fail_at) return 2; *p = malloc(n); return 0; }
static int cudaFree(void* p) { free(p); return 0; }
static int cudaGetLastError() { return 0; }
%s
static sph_ctx c;
// sets the context up, fails allocation `at` of the first call; a second call with
// none failing: r[0], r[1] the two results, r[2] whether every buffer is there
extern "C" void run(int at, int again_fails, int* r) {
  c = sph_ctx();
  for (int f = 0; f < 5; f++) c.nf[f] = 40;
  c.N = 40;
  calls = 0; fail_at = at;
  r[0] = adj_alloc(&c, 2);
  calls = 0; fail_at = again_fails;
  r[1] = adj_alloc(&c, 2);
  r[2] = c.adjS && c.adjW && c.adjC && c.adjK >= 2;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    with open(os.path.join(CSRC, "sph.cu")) as f:
        body = re.search(r"^static int adj_alloc\(.*?^}\n", f.read(), re.S | re.M).group(0)
    d = tmp_path_factory.mktemp("adj_alloc")
    src, lib = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS % body)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    run = ctypes.CDLL(str(lib)).run

    def call(at, again_fails):
        r = (ctypes.c_int * 3)()
        run(at, again_fails, r)
        return list(r)
    return call


def test_all_allocations_succeed(harness):
    assert harness(0, 0) == [0, 0, 1]


@pytest.mark.parametrize("at", [1, 2, 3])
def test_second_call_after_a_failure(harness, at):
    assert harness(at, 0) == [-5, 0, 1]
    first, second, whole = harness(at, 1)
    assert first == -5 and second == -5 and not whole
