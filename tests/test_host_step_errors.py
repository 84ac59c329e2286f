"""The host-fed step's errors, without a GPU: csrc/host_step.cu linked against a fake of the CUDA runtime that knows which work is ordered
behind which, and in which every call fails in turn.  Whatever fails, the call says so, the caller's stream ends behind every copy
that was enqueued on the side streams, and no stream is waited for that does not hang on the caller's (which would break a
capture)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_21911_b200", "csrc")

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <vector>
#include "sv.h"

static int calls, fail_at, violations;
static bool pinned, failed_joining;
static int next_op;
struct Event { std::set<int> ops; int from = -1; };
static std::vector<Event> events;
static std::set<int> stream_ops[4];        // streams 1 (the caller's), 2 (uploads), 3 (downloads)
static bool forked[4];
static std::set<int> side_ops;             // copies on the side streams
static std::vector<std::vector<int>> uploads_of, compute_of;
static int id(cudaStream_t s) { return (int)(size_t)s; }
static bool fails() { return calls++ == fail_at; }
static int enqueue(int s) { stream_ops[s].insert(next_op); if (s > 1) side_ops.insert(next_op); return next_op++; }

extern "C" {
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { events.emplace_back(); *e = (cudaEvent_t)events.size(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *at, const void *p)
{
    memset(at, 0, sizeof *at);
    at->type = pinned ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    at->devicePointer = const_cast<void *>(p);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    if (fails()) { failed_joining = (size_t)e == 2; return cudaErrorUnknown; }
    if (id(s) > 1 && !forked[id(s)]) ++violations, printf("stream %d is recorded without hanging on the caller's\n", id(s));
    events[(size_t)e - 1].ops = stream_ops[id(s)];
    events[(size_t)e - 1].from = id(s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    if (fails()) { failed_joining = (size_t)e == 2; return cudaErrorUnknown; }
    Event &ev = events[(size_t)e - 1];
    stream_ops[id(s)].insert(ev.ops.begin(), ev.ops.end());
    if (ev.from == 1) forked[id(s)] = true;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t s)
{
    if (fails()) return cudaErrorUnknown;
    if (!forked[id(s)]) ++violations, printf("a copy on stream %d is not behind the caller's work\n", id(s));
    enqueue(id(s));
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *, void **)
{
    if (fails()) return cudaErrorUnknown;
    enqueue(id(cfg->stream));
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorUnknown; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
char __cudaInitModule(void **) { return 1; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }

static sv_status work(void *s)
{
    if (fails()) return SV_ERR_SHAPE;
    enqueue(id((cudaStream_t)s));
    return SV_OK;
}
sv_status sv_block_reps_layers(const sv_geom *, const sv_layers *, const uint8_t *, int32_t, int32_t, float *, void *s) { return work(s); }
sv_status sv_select_blocks_layers(const sv_geom *, const sv_layers *, int32_t, int32_t, const uint8_t *, const void *, const float *,
                                  const int32_t *, int32_t, int32_t, int32_t *, int32_t *, int32_t, void *s) { return work(s); }
}
namespace svh {
sv_status verify_attn_layers(const sv_geom *, const sv_layers *, int32_t, int32_t, const uint8_t *, const void *, const void *,
                             const void *, const int32_t *, const int32_t *, const int32_t *, int32_t, float, void *, void *,
                             size_t, int32_t *, void *s, bool) { return work(s); }
}

int main()
{
    alignas(128) static char mem[1 << 16];
    int runs = 0, bad = 0;
    for (int p = 0; p < 2; ++p)
        for (int n_chunks = 1; n_chunks <= 4; ++n_chunks)
            for (int at = -1;; ++at) {
                events.clear();
                sv_host_step *h = sv_host_step_create();
                pinned = p == 0, calls = 0, fail_at = at, failed_joining = false, violations = 0, next_op = 0;
                for (auto &o : stream_ops) o.clear();
                forked[1] = true, forked[2] = forked[3] = false;
                side_ops.clear();
                const sv_geom g = {1, 2, 1, 128, 64, 1, 1};
                const sv_layers layers = {mem, (int32_t *)mem, (int32_t *)mem, 4};
                const int32_t ends[4][4] = {{4}, {1, 4}, {1, 3, 4}, {1, 2, 3, 4}};
                const uint8_t anchors[4] = {1, 1, 1, 1};
                const sv_status st = sv_verify_step_from_host(
                    h, &g, &layers, anchors, ends[n_chunks - 1], n_chunks, mem, mem, mem, mem, mem, mem, nullptr, (float *)mem, (int32_t *)mem,
                    1, 1, (int32_t *)mem, (int32_t *)mem, 4, mem, mem, mem, sizeof mem, nullptr, 1, nullptr, (void *)2, (void *)3, (void *)1);
                const bool failed = at >= 0 && calls > at;
                int loose = 0;
                for (int op : side_ops) loose += !stream_ops[1].count(op);
                const bool wrong = (st == SV_OK) == failed || violations || (loose && !failed_joining);
                if (wrong) printf("%s, %d chunks, call %d of %d fails: status %d, %d copies not joined\n", p ? "pageable" : "pinned", n_chunks, at, calls, (int)st, loose);
                bad += wrong, ++runs;
                sv_host_step_destroy(h);
                if (at >= 0 && !failed) break;   // (every call has failed once)
            }
    printf("%d runs\n", runs);
    return bad != 0 || runs < 100;
}
"""


def test_every_call_fails_in_turn(tmp_path):
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    (tmp_path / "fake.cpp").write_text(FAKE)
    obj, exe = str(tmp_path / "host_step.o"), str(tmp_path / "run")
    inc = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", *inc, "-c", os.path.join(CSRC, "host_step.cu"), "-o", obj], check=True)
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.run(["g++", "-std=c++17", *inc, "-I", cuda, str(tmp_path / "fake.cpp"), obj, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
