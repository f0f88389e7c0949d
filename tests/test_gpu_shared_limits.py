"""A kernel's limit of dynamic shared memory belongs to the kernel, not to a
handle: a call that needs less of it must not refuse the launch of another
handle or thread that needs more.  Two batches on one kernel with different
horizons, stepped in turn, and two host threads that project sequences of
different lengths at the same time."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"

THREADS = r"""
#include <pthread.h>
typedef int (*fn_t)(int, int, float, const float*, int, float, const float*, const float*, const float*, const float*,
                    float*, void*);
struct job { fn_t fn; int H, calls, bad; const float *b, *q; float* v; void* s; };
static void* run(void* p) {
    struct job* j = (struct job*)p;
    for (int i = 0; i < j->calls; ++i)
        j->bad += j->fn(1, j->H, 0.01f, j->b, 0, 1.0f, 0, j->q, j->q, j->v, j->v, j->s) != 0;
    return 0;
}
int both(fn_t fn, int H0, int H1, const float* b, const float* q, float* v0, float* v1, void* s0, void* s1, int calls) {
    struct job a = {fn, H0, calls, 0, b, q, v0, s0}, c = {fn, H1, calls, 0, b, q, v1, s1};
    pthread_t t;
    if (pthread_create(&t, 0, run, &c)) return -1;
    run(&a);
    pthread_join(t, 0);
    return a.bad + c.bad;
}
"""


@pytest.mark.parametrize("cfg,K,lps,spc", [(3, 2500, 16, 16), (1, 2500, 16, 16), (2, 64, 32, 8), (1, 64, 8, 32)])
def test_batches_of_different_horizons_step_in_turn(tmp_path, monkeypatch, cfg, K, lps, spc):
    monkeypatch.setenv("MPPI_TUNE_FILE", str(tmp_path / "none.txt"))
    from paper_2511_21264_gb300 import native
    sc = scenes.config(cfg)
    m = native.Model(sc.to_blob())
    x = torch.tensor(m.home(), device=DEV)
    batches, us = [], []
    for H in (24, 3):  # the second one needs less
        b = native.Batch([(m, K, H, 1.0, sc.sigma_vec(), 5), (m, K, H, 1.0, sc.sigma_vec(), 6)])
        b.set_launch(1, 1)
        b.set_layout(lps, 0)
        b.set_launch(spc, 1)
        batches.append(b)
        us.append([torch.zeros((H, sc.nu), device=DEV) for _ in range(2)])
    for b, u in list(zip(batches, us)) * 2:
        b.step([x, x], u)
        assert b.sync()[0] == 0
    assert all(torch.isfinite(u).all() and u.abs().max() > 0 for pair in us for u in pair)


@pytest.mark.parametrize("H0,H1", [(100, 128), (200, 128)])
def test_projections_of_two_threads(tmp_path, H0, H1):
    from paper_2511_21264_gb300 import native
    src, so = tmp_path / "threads.c", tmp_path / "threads.so"
    src.write_text(THREADS)
    subprocess.run(["gcc", "-O2", "-shared", "-fPIC", "-o", os.fspath(so), os.fspath(src), "-lpthread"], check=True)
    p = C.c_void_p
    b = np.array([-1, 1, -3, 3, -10, 10, -300, 300], np.float32)
    q, v = torch.zeros(1, device=DEV), torch.zeros((2, 256), device=DEV)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    refused = C.CDLL(os.fspath(so)).both(C.cast(native.lib().mppi_qp_project, p), H0, H1, p(b.ctypes.data),
                                         p(q.data_ptr()), p(v[0].data_ptr()), p(v[1].data_ptr()),
                                         p(streams[0].cuda_stream), p(streams[1].cuda_stream), 10000)
    torch.cuda.synchronize()
    assert refused == 0
