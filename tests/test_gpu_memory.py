"""Device memory that runs out: the library's objects are linked here with a cudaMalloc and a
cudaMallocAsync that fail when they are told to (an error code; nothing goes wrong on the
device), and child processes check what is left. A batch whose members change form builds its
groups again inside a run; a failed attempt leaves it as usable as before. An instance whose
column form's words do not fit is made without them and runs row by row."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = """
#include <stddef.h>
extern int __real_cudaMalloc(void **p, size_t n);
static int left = -1;
void fail_cuda_malloc(int calls) { left = calls; }
int __wrap_cudaMalloc(void **p, size_t n)
{
    if (left >= 0 && left-- == 0) {
        *p = NULL;
        return 2; /* cudaErrorMemoryAllocation */
    }
    return __real_cudaMalloc(p, n);
}
extern int __real_cudaMallocAsync(void **p, size_t n, void *stream);
static int left_async = -1;
void fail_cuda_malloc_async(int calls) { left_async = calls; }
int __wrap_cudaMallocAsync(void **p, size_t n, void *stream)
{
    if (left_async >= 0 && left_async-- == 0) {
        *p = NULL;
        return 2;
    }
    return __real_cudaMallocAsync(p, n, stream);
}
"""


def run_child(tmp_path, what):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30862_gb300 import build as B
    src, obj, lib = (str(tmp_path / n) for n in ("fake.c", "fake.o", "libqieo.so"))
    with open(src, "w") as fh:
        fh.write(FAKE)
    subprocess.check_call(["gcc", "-O1", "-fPIC", "-c", src, "-o", obj])
    B.link(lib, obj, "-Xlinker", "--wrap=cudaMalloc", "-Xlinker", "--wrap=cudaMallocAsync")
    r = subprocess.run([sys.executable, os.path.abspath(__file__), lib, what], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


@pytest.mark.gpu
def test_a_failed_regrouping_leaves_no_groups(tmp_path):
    assert run_child(tmp_path, "regroup").count("regrouped") == 3


@pytest.mark.gpu
def test_an_instance_without_room_for_the_column_form(tmp_path):
    assert run_child(tmp_path, "instance").count("solved") == 2


def child(lib, what):
    sys.path[:0] = [ROOT, os.path.dirname(os.path.abspath(__file__))]
    from oracle import oracle as O
    from paper_2609_30862_gb300 import build as B
    from paper_2609_30862_gb300 import qieo as Q
    from paper_2609_30862_gb300 import workload as W
    from saturated import load_state
    B.LIB = lib
    Q.load(build_if_missing=False)
    fake = ctypes.CDLL(lib)
    prob, np_ = W.knapsack(1500, 8), 40
    if what == "instance":
        ref = O.run(prob, np_, 40, seed=1)
        fake.fail_cuda_malloc_async(0)
        with Q.Instance(prob, np_, seed=1) as I, Q.Instance(prob, np_, seed=1) as J:
            for _ in range(2):         # alone, and in a batch beside one that has the words
                I.run(25)
                with Q.Batch([I, J]) as b:
                    b.run(15)
                k, t = I.state()
                assert t == 40 and np.array_equal(k, ref.k) and np.array_equal(I.history(0, 40)[0], ref.hist_e)
                assert np.array_equal(I.alleles(), ref.x) and np.array_equal(I.best()[0], ref.best_x)
                I.reset()
                print("solved")
        return
    k0 = np.random.default_rng(3).integers(-25, 26, size=(np_, 1500)).astype(np.int16)
    st = O.State(np_, prob.ng)
    st.k[:] = k0
    refs = [O.run(prob, np_, 30, seed=1, state=st), O.run(prob, np_, 30, seed=2), O.run(prob, np_, 30, seed=3, rule=1)]
    insts = [Q.Instance(prob, np_, seed=i + 1, rule=1 if i == 2 else 0) for i in range(3)]
    with Q.Batch(insts) as b:
        for failing in range(3):       # a group of its own for each member once the first changed form
            for I in insts:
                I.reset()
            b.run(3)                   # all rule R1 members in the column form
            for I in insts:
                I.reset()
            load_state(insts[0], k0)
            fake.fail_cuda_malloc(failing)
            try:
                b.run(30)
            except Q.QieoError as e:
                assert e.status == Q.QIEO_ERR_OOM, e
            else:
                raise AssertionError("the allocation did not fail")
            b.run(30)
            for I, ref in zip(insts, refs):
                k, t = I.state()
                assert t == 30 and np.array_equal(k, ref.k)
                assert np.array_equal(I.history(0, 30)[0], ref.hist_e)
                assert np.array_equal(I.alleles(), ref.x) and np.array_equal(I.best()[0], ref.best_x)
            print("regrouped")
    for I in insts:
        I.close()


if __name__ == "__main__":
    child(*sys.argv[1:])
