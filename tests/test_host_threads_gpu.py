"""Scores of different sizes from two host threads on two streams at once, through the C ABI: every call
is enqueued, and its result is that of the same call alone.  (A kernel's limit on dynamic shared memory
belongs to the function: a launch that sets its own size can take the room from the other thread's.)"""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ROUNDS, CALLS = 150, 40          # the stream is waited for after every CALLS calls

PROGRAM = r"""
#include <pthread.h>
#include "vqnnf.h"

typedef struct {
    const uint8_t *lab; int H, W, k, th, tw; const vqnnf_filter *bank; int F; const int32_t *tc;
    float *heat; int32_t *am; void *ws; size_t ws_bytes; void *stream; int rounds, calls, failed;
} job;

static pthread_barrier_t start;

static void *work(void *p)
{
    job *j = (job *)p;
    pthread_barrier_wait(&start);
    for (int r = 0; r < j->rounds; ++r) {
        for (int c = 0; c < j->calls; ++c)
            j->failed += vqnnf_score(j->lab, j->H, j->W, j->k, j->th, j->tw, j->bank, j->F, j->tc, j->heat, j->am,
                                     j->ws, j->ws_bytes, j->stream) != VQNNF_OK;
        j->failed += vqnnf_last_device_error(j->stream) != VQNNF_OK;
    }
    return 0;
}

int together(job *a, job *b)
{
    pthread_t t;
    if (pthread_barrier_init(&start, 0, 2) || pthread_create(&t, 0, work, b)) return 1;
    work(a);
    pthread_join(t, 0);
    pthread_barrier_destroy(&start);
    return 0;
}
"""


class Job(ctypes.Structure):
    _fields_ = [("lab", ctypes.c_void_p)] + [(n, ctypes.c_int) for n in ("H", "W", "k", "th", "tw")] + \
        [("bank", ctypes.c_void_p), ("F", ctypes.c_int)] + \
        [(n, ctypes.c_void_p) for n in ("tc", "heat", "am", "ws")] + [("ws_bytes", ctypes.c_size_t), ("stream", ctypes.c_void_p)] + \
        [(n, ctypes.c_int) for n in ("rounds", "calls", "failed")]


@pytest.fixture(scope="module")
def vq():
    from paper_2306_15010_gb300 import build
    build.build()
    import paper_2306_15010_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.fixture(scope="module")
def together(vq, tmp_path_factory):
    cc = shutil.which("gcc") or pytest.skip("no C compiler")
    d = tmp_path_factory.mktemp("threads")
    (d / "t.c").write_text(PROGRAM)
    lib = os.path.join(ROOT, "paper_2306_15010_gb300")
    r = subprocess.run([cc, "-std=gnu99", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-pthread", "-I", os.path.join(ROOT, "include"),
                        str(d / "t.c"), "-L", lib, "-lvqnnf", f"-Wl,-rpath,{lib}", "-o", str(d / "t.so")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(d / "t.so")).together


def test_two_threads(vq, together):
    # the strip counts of a row of labels, 4 k bytes per 64 columns: 33 and 67 KB
    H, k, th, tw = 33, 256, 30, 32
    jobs, keep = [], []
    for W in (2000, 4100):
        g = torch.Generator().manual_seed(W)
        lab = torch.randint(0, k, (H, W), generator=g).to(torch.uint8).cuda()
        bank = vq.Bank(synth.grid_bank(th, tw, 2))
        tc = vq.vqnnf_filter_responses(lab[:th, :tw].contiguous(), k, bank)
        ws = vq.Workspace(vq.vqnnf_workspace_bytes(3, H, W, 0, k, th, tw, bank.F))
        heat, am = vq.vqnnf_score(lab, k, th, tw, bank, tc, ws=ws)
        alone = heat.clone()
        stream = torch.cuda.Stream()
        jobs.append(Job(lab.data_ptr(), H, W, k, th, tw, bank.ptr, bank.F, tc.data_ptr(), heat.data_ptr(), am.data_ptr(),
                        ws.ptr, ws.nbytes, stream.cuda_stream, ROUNDS, CALLS, 0))
        keep.append((lab, bank, tc, ws, heat, alone, am, stream))
    torch.cuda.synchronize()
    for _, _, _, _, heat, _, _, _ in keep:
        heat.zero_()
    torch.cuda.synchronize()
    assert together(ctypes.byref(jobs[0]), ctypes.byref(jobs[1])) == 0
    torch.cuda.synchronize()
    assert [j.failed for j in jobs] == [0, 0]
    for _, _, _, _, heat, alone, _, _ in keep:
        assert torch.equal(heat, alone)
