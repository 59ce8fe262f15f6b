// Stands in for the CUDA runtime and for the kernel launchers under csrc/api.cu: every call is written to a log and succeeds, or fails where
// fake_reset says so.  Nothing runs; the tests read the order in which work was enqueued.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <cstdlib>
#include <string>

#include "molora.h"

namespace {
std::string g_log, g_fail_name;
int g_fail_at = -1, g_priority = 0;
uintptr_t g_next = 0x100;
bool note(const char* name, const std::string& rest)
{
    g_log += std::string(name) + " " + rest + "\n";
    return !(g_fail_name == name && g_fail_at-- == 0);
}
std::string num(const void* p) { return std::to_string(reinterpret_cast<uintptr_t>(p)); }
cudaError_t done(bool ok) { return ok ? cudaSuccess : cudaErrorUnknown; }
molora_status_t launched(const char* name, const molora_proj_desc_t* projs, int32_t P, int64_t N, const void* ws, cudaStream_t s)
{
    std::string rest = num(s) + " " + std::to_string(N) + " " + num(ws);
    for (int i = 0; i < P; ++i) rest += " " + num(projs[i].x) + " " + std::to_string(projs[i].d_in) + " " + num(projs[i].y) + " " + std::to_string(projs[i].d_out);
    return note(name, rest) ? MOLORA_OK : MOLORA_ERR_CUDA;
}
}  // namespace

extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_reset(const char* fail_name, int fail_at, int priority)
{
    g_log.clear();
    g_fail_name = fail_name;
    g_fail_at = fail_at;
    g_priority = priority;
}
void fake_report_at_exit()                     // what is called from here on, printed when the process ends
{
    g_log.clear();
    std::atexit([] {
        std::printf("%send\n", g_log.c_str());
        std::fflush(stdout);
    });
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t s)
{
    return done(note(kind == cudaMemcpyHostToDevice ? "upload" : "download", num(s) + " " + num(dst) + " " + num(src) + " " + std::to_string(n)));
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    *s = reinterpret_cast<cudaStream_t>(g_next++);
    return done(note("stream", num(*s) + " 0"));
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int priority)
{
    *s = reinterpret_cast<cudaStream_t>(g_next++);
    return done(note("stream", num(*s) + " " + std::to_string(priority)));
}
cudaError_t cudaStreamGetPriority(cudaStream_t, int* priority)
{
    *priority = g_priority;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return done(note("destroy_stream", num(s))); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned)
{
    *e = reinterpret_cast<cudaEvent_t>(g_next++);
    return done(note("event", num(*e)));
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return done(note("destroy_event", num(e))); }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return done(note("record", num(s) + " " + num(e))); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return done(note("wait", num(s) + " " + num(e))); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c)
{
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int)
{
    *v = 148;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}

namespace molora {
// (widths are multiples of 64 in the tests)
bool decode_eligible(const molora_proj_desc_t& p, molora_dtype_t dt) { return dt == MOLORA_BF16 && p.rank >= 16 && p.d_in % 32 == 0 && p.d_out % 32 == 0; }
bool stream_eligible(const molora_proj_desc_t& p, molora_dtype_t dt) { return decode_eligible(p, dt); }
bool umma_eligible(const molora_proj_desc_t& p, molora_dtype_t dt) { return decode_eligible(p, dt); }
bool jobs_eligible(const molora_proj_desc_t& p, molora_dtype_t dt, int64_t N) { return decode_eligible(p, dt) && N <= 1024; }
bool group_apply_umma_eligible(int64_t N, int32_t) { return N <= 4096; }
bool group_apply_stream_eligible(int64_t N) { return N <= 4096; }
bool group_apply_decode_eligible(int64_t N) { return N <= 1024; }
bool group_apply_rowtile_eligible(const molora_proj_desc_t*, int32_t, molora_dtype_t, int64_t, int32_t) { return false; }
size_t jobs_control_bytes() { return 256; }
size_t jobs_partial_bytes(int64_t N, int32_t, int32_t d_in, int32_t rank) { return (size_t)N * rank * (d_in / 512 + 1) * 4; }
size_t decode_workspace_bytes(int64_t N, int32_t d_in, int32_t rank) { return (size_t)N * rank * (d_in / 256 + 1) * 4; }
size_t group_workspace_bytes(int64_t, int32_t) { return 0; }
size_t route_gate_workspace_bytes(molora_dtype_t, int32_t, int32_t) { return 256; }
size_t route_gate_prepared_workspace_bytes(molora_dtype_t, int32_t, int32_t) { return 256; }
size_t route_mlp_workspace_bytes(molora_dtype_t, int32_t, int32_t) { return 256; }

molora_status_t launch_group(const int32_t*, int64_t N, int32_t, int32_t*, int32_t*, int32_t*, void*, size_t, uint32_t*, cudaStream_t s)
{
    return launched("group", nullptr, 0, N, nullptr, s);
}
molora_status_t launch_route_gate(const void*, molora_dtype_t, int64_t N, int32_t, int64_t, const float*, const float*, int32_t, int32_t*, float*,
                                  void*, uint32_t*, cudaStream_t s, int)
{
    return launched("route", nullptr, 0, N, nullptr, s);
}
molora_status_t launch_route_vocab(const int32_t*, int64_t N, const int32_t*, int32_t, const int32_t*, int32_t, int32_t*, uint32_t*, cudaStream_t s,
                                   const int32_t*, int32_t)
{
    return launched("route", nullptr, 0, N, nullptr, s);
}
molora_status_t launch_apply_umma(const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, const int32_t*, const int32_t*, uint32_t*, int32_t,
                                  cudaStream_t s, const int32_t*, int32_t*, int32_t, int32_t, const uint8_t*)
{
    return launched("apply", p, P, N, nullptr, s);
}
molora_status_t launch_apply_stream(const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, const int32_t*, const int32_t*, int32_t, uint32_t*,
                                    cudaStream_t s)
{
    return launched("apply", p, P, N, nullptr, s);
}
molora_status_t launch_group_apply_stream(const int32_t*, const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, int32_t*, int32_t*, int32_t*,
                                          uint32_t*, cudaStream_t s)
{
    return launched("apply", p, P, N, nullptr, s);
}
molora_status_t launch_apply_decode(const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, const int32_t*, const int32_t*, int32_t, void* ws,
                                    size_t, uint32_t*, cudaStream_t s)
{
    return launched("apply_pair", p, P, N, ws, s);
}
molora_status_t launch_group_apply_decode(const int32_t*, const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, int32_t*, int32_t*, int32_t*,
                                          void* ws, size_t, uint32_t*, cudaStream_t s)
{
    return launched("apply_pair", p, P, N, ws, s);
}
molora_status_t launch_apply_jobs(const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, const int32_t*, const int32_t*, void* ctl, void*, size_t,
                                  uint32_t*, cudaStream_t s)
{
    return launched("apply_jobs", p, P, N, ctl, s);
}
molora_status_t launch_group_apply_jobs(const int32_t*, const molora_proj_desc_t* p, int32_t P, int64_t N, int32_t, int32_t*, int32_t*, int32_t*,
                                        void* ctl, void*, size_t, uint32_t*, cudaStream_t s)
{
    return launched("apply_jobs", p, P, N, ctl, s);
}
molora_status_t launch_apply_rowtile(const molora_proj_desc_t* p, int32_t P, molora_dtype_t, int64_t N, int32_t, const int32_t*, const int32_t*,
                                     int32_t, cudaStream_t s)
{
    return launched("apply", p, P, N, nullptr, s);
}
// never reached by the tests
molora_status_t launch_route_mlp(const void*, molora_dtype_t, int64_t, int32_t, int64_t, const float*, const float*, int32_t, const float*, const float*,
                                 int32_t, int32_t*, float*, void*, size_t, uint32_t*, cudaStream_t, int) { return MOLORA_ERR_CUDA; }
molora_status_t launch_topk_sets(const int32_t*, const float*, int64_t, int32_t, int32_t, int32_t*, float*, uint8_t*, cudaStream_t) { return MOLORA_ERR_CUDA; }
molora_status_t launch_topk_softmax(const float*, int64_t, int32_t, int32_t, int32_t*, float*, cudaStream_t) { return MOLORA_ERR_CUDA; }
molora_status_t launch_group_apply_rowtile(const int32_t*, const molora_proj_desc_t*, int32_t, molora_dtype_t, int64_t, int32_t, int32_t*, int32_t*,
                                           int32_t*, uint32_t*, cudaStream_t) { return MOLORA_ERR_CUDA; }
molora_status_t launch_apply_stream_sets(const molora_proj_desc_t*, int32_t, int64_t, int32_t, int32_t, int32_t, const uint8_t*, const int32_t*,
                                         const int32_t*, uint32_t*, cudaStream_t) { return MOLORA_ERR_CUDA; }
molora_status_t launch_group_apply_stream_sets(const int32_t*, const molora_proj_desc_t*, int32_t, int64_t, int32_t, int32_t, int32_t, const uint8_t*,
                                               int32_t*, int32_t*, int32_t*, uint32_t*, cudaStream_t) { return MOLORA_ERR_CUDA; }
molora_status_t launch_bounded_wait_selftest(uint32_t*, int64_t, int32_t*, cudaStream_t) { return MOLORA_ERR_CUDA; }
}  // namespace molora
