"""What the library asks of the CUDA runtime, seen and steered by a shim in front
of libcudart: limits of a kernel that all plans of a process share, and calls
that fail.  The shim is preloaded into a child process, once for all tests."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <cuda_runtime_api.h>

static void* find(const char* name) {
    void* f = dlsym(RTLD_NEXT, name);   /* where libcudart is in the global scope */
    return f ? f : dlsym(dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD), name);
}
#define REAL(f) __typeof__(&f) real = (__typeof__(&f))find(#f)

/* limits: how often a kernel's shared memory was set below an earlier value */
static const void* funcs[1024];
static int values[1024], nfuncs, lowered, last_errors;
int shim_lowered(void) { return lowered; }
int shim_last_errors(void) { return last_errors; }

cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
    REAL(cudaFuncSetAttribute);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        int k = 0;
        while (k < nfuncs && funcs[k] != f) ++k;
        if (k == nfuncs && nfuncs < 1024) {
            funcs[nfuncs++] = f;
            values[k] = v;
        }
        if (k < nfuncs) {
            if (v < values[k]) ++lowered;
            values[k] = v;
        }
    }
    return real(f, a, v);
}

cudaError_t cudaGetLastError(void) {
    REAL(cudaGetLastError);
    ++last_errors;
    return real();
}

/* allocations of this many bytes and more fail (0: none) */
static size_t fail_from;
void shim_fail_malloc_from(size_t bytes) { fail_from = bytes; }
cudaError_t cudaMalloc(void** p, size_t bytes) {
    REAL(cudaMalloc);
    return fail_from && bytes >= fail_from ? cudaErrorMemoryAllocation : real(p, bytes);
}

/* clusters: a size whose query fails, and the last one launched */
static unsigned refused, launched;
void shim_refuse_cluster(unsigned blocks) { refused = blocks; }
unsigned shim_launched_cluster(void) { return launched; }
static unsigned cluster_of(const cudaLaunchConfig_t* c) {
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension)
            return c->attrs[k].val.clusterDim.x;
    return 1;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    REAL(cudaOccupancyMaxActiveClusters);
    return refused && cluster_of(c) == refused ? cudaErrorInvalidClusterSize : real(n, f, c);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    REAL(cudaLaunchKernelExC);
    launched = cluster_of(c);
    return real(c, f, args);
}
"""

CHILD = r"""
import ctypes, json, sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import torch
import synth
from gpu_util import dev, plan_for

shim = ctypes.CDLL(sys.argv[2])
shim.shim_fail_malloc_from.argtypes = [ctypes.c_size_t]
out = {}


def rhs(A):
    return torch.tensor(synth.uniform(A.n, 7), device=dev())


def one_block():
    big, small = synth.lap2d_5pt_lower(60, 450), synth.lap2d_5pt_lower(60, 150)
    with plan_for(big) as p, plan_for(small) as q:
        for plan, A in ((p, big), (q, small), (p, big)):
            plan.set_tuning(2, 256, 0)
            plan.solve(rhs(A))
            assert plan.last_launch_count == 1      # the one-block kernel
    out["lowered"] = shim.shim_lowered()


def cluster():
    A = synth.general_lower(4000, 5)
    b = rhs(A)
    with plan_for(A) as p:
        p.set_tuning(32, 256, 0)
        want = p.solve(b, algo="blocked")
        p.solve(b)
        out["cluster_first"] = [p.last_launch_count, shim.shim_launched_cluster()]
        counts = []
        for _ in range(2):
            before = shim.shim_last_errors()
            p.solve(b)
            counts.append(shim.shim_last_errors() - before)
    with plan_for(A) as p:                          # a plan that has not asked yet
        p.set_tuning(32, 256, 0)
        before = shim.shim_last_errors()
        p.solve(b)
        out["last_errors"] = [shim.shim_last_errors() - before, counts[1]]
    shim.shim_refuse_cluster(16)
    with plan_for(A) as p:
        p.set_tuning(32, 256, 0)
        got = p.solve(b)
        out["cluster_refused"] = [p.last_launch_count, shim.shim_launched_cluster(),
                                  bool(torch.equal(got, want))]
    shim.shim_refuse_cluster(0)


def no_room():
    A = synth.lap3d_7pt_ilu0(40, 41, 43)[0]
    b = rhs(A)
    with plan_for(A) as p, plan_for(A) as q:
        for plan in (p, q):
            plan.set_tuning(8, 256, 0)              # twice as many slots as entries
            plan.best_algo = "partitioned"
        want, _, _ = p.solve_refined(b)
        q.solve(b, algo="partitioned")              # its FP64 copy is there
        shim.shim_fail_malloc_from(6 * A.nnz)       # room for nnz floats, not for the slices
        try:
            got, _, _ = q.solve_refined(b)
            out["refined"] = bool(torch.equal(got, want))
        except Exception as e:
            out["refined"] = repr(e)
        shim.shim_fail_malloc_from(0)


for f in (one_block, cluster, no_room):
    f()
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def seen(cuda_device, tmp_path_factory):
    from paper_1710_04985_gb300 import build
    d = tmp_path_factory.mktemp("shim")
    (d / "shim.c").write_text(SHIM)
    (d / "child.py").write_text(CHILD)
    inc = os.path.join(os.path.dirname(build._cuda_lib_dir(build._nvcc())), "include")
    so = str(d / "shim.so")
    r = subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", inc, str(d / "shim.c"), "-o", so,
                        "-ldl"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([sys.executable, str(d / "child.py"), ROOT, so], capture_output=True,
                       text=True, timeout=300, env=dict(os.environ, LD_PRELOAD=so))
    assert r.returncode == 0, r.stdout + r.stderr
    return json.loads(r.stdout.splitlines()[-1])


def test_one_block_solves_never_lower_the_limit_of_another_plan(seen):
    """The limit belongs to the kernel, not to the plan: a smaller system must not
    take away what a larger one, launched by another thread, is about to use."""
    assert seen["lowered"] == 0


def test_a_cluster_size_that_cannot_be_asked_for_leaves_the_smaller_one(seen):
    assert seen["cluster_first"] == [1, 16]
    assert seen["cluster_refused"] == [1, 8, True]


def test_asking_for_the_cluster_size_clears_no_error_of_the_caller(seen):
    first, later = seen["last_errors"]
    assert first == later


def test_refined_solve_without_room_for_the_fp32_slices(seen):
    assert seen["refined"] is True


def test_two_threads_with_plans_of_their_own(cuda_device):
    """The calls of both are valid whatever the other one launches in between."""
    import threading

    import torch

    import synth
    from gpu_util import dev, plan_for
    errors = []

    def work(ny):
        try:
            A = synth.lap2d_5pt_lower(60, ny)
            b = torch.tensor(synth.uniform(A.n, 7), device=dev())
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), plan_for(A) as p:
                p.set_tuning(2, 256, 0)
                want = p.solve(b, algo="blocked")
                x = torch.empty_like(b)
                for _ in range(300):
                    p.solve(b, out=x)
                stream.synchronize()
                assert torch.equal(x, want)
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(ny,)) for ny in (450, 150)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
