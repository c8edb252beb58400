"""Groups on side streams when a call fails, on a fake of the CUDA runtime: the stream
that goes on is ordered after all work that was queued, whichever call failed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#pragma once
#include <map>
#include <vector>
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 999 };
struct FakeStream { int queued = 0, synced = 0; std::map<FakeStream *, int> after; };
struct FakeEvent { FakeStream *s = nullptr; int at = 0; };
typedef FakeStream *cudaStream_t;
typedef FakeEvent *cudaEvent_t;
enum { cudaEventDisableTiming = 2, cudaStreamNonBlocking = 1 };
inline int g_calls = 0, g_fail_at = -1;  // the call that fails
inline bool fails() { return g_calls++ == g_fail_at; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, int) { if (fails()) return cudaErrorUnknown; *s = new FakeStream; return cudaSuccess; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, int) { if (fails()) return cudaErrorUnknown; *e = new FakeEvent; return cudaSuccess; }
inline cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
inline cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { if (fails()) return cudaErrorUnknown; e->s = s; e->at = s->queued; return cudaSuccess; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, int) { if (fails()) return cudaErrorUnknown; s->after[e->s] = e->at; return cudaSuccess; }
inline cudaError_t cudaStreamSynchronize(cudaStream_t s) { s->synced = s->queued; return cudaSuccess; }
"""

MAIN = r"""
#include <cstdio>
#include "side_streams.h"
int main() {
    int bad = 0, runs = 0;
    for (int own = 0; own < 8; ++own)              // which of three groups have a side stream
        for (int warm = 0; warm < 2; ++warm)       // streams made by an earlier run or by this one
            for (int fail = -1; fail < 24; ++fail, ++runs) {
                qsg::SideStreams side;
                FakeStream st;
                std::vector<cudaStream_t> used;
                auto run = [&] {
                    return side.run(
                        3, &st, [&](size_t i) { return (own >> i & 1) != 0; },
                        [&](size_t, cudaStream_t t) {
                            ++t->queued;                        // a launch goes out,
                            used.push_back(t);
                            const bool f = fails();             // the next one may fail
                            if (!f) ++t->queued;
                            return f ? QSG_ERR_ARG : QSG_OK;
                        },
                        [](cudaError_t) { return QSG_ERR_CUDA; });
                };
                g_fail_at = -1;
                if (warm && run() != QSG_OK) ++bad;
                used.clear();
                g_calls = 0;
                g_fail_at = fail;
                const qsg_status s = run();
                if ((s != QSG_OK) != (fail >= 0 && fail < g_calls)) ++bad;
                for (cudaStream_t t : used)
                    if (t != &st && st.after[t] < t->queued && t->synced < t->queued) {
                        std::printf("own %d warm %d fail %d: work queued after the join\n", own, warm, fail);
                        ++bad;
                    }
            }
    std::printf("%d runs\n", runs);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_every_failure_still_joins_the_streams(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    cmd = ["g++", "-std=c++17", "-I", str(tmp_path), "-I", os.path.join(ROOT, "include"), "-I",
           os.path.join(ROOT, "paper_2310_07486_gb300", "csrc"), str(tmp_path / "main.cpp"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    assert "400 runs" in r.stdout
