// Shared device/host helpers for the sm_103a kernels of the HQS hot path.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hqs.h"

#define HQS_DEV __device__ __forceinline__

// ---------------------------------------------------------------- complex
// Complex add and subtract as one packed FP32x2 instruction each (sm_100 and later; every
// component rounded to nearest as by the scalar instruction).  The transform passes are
// bound by instruction issue: A^H A at 320^2 x 16 coils 51.1 -> 49.8 us, the one-slice
// solve step 788 -> 750 us, the volume solve 1883 -> 1762 us.
HQS_DEV float2 cadd(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 p, q, s;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\t"
        "add.rn.f32x2 s, p, q;\n\tmov.b64 {%0, %1}, s;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
HQS_DEV float2 csub(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 p, q, s;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\t"
        "sub.rn.f32x2 s, p, q;\n\tmov.b64 {%0, %1}, s;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// acc + a s and a s for a real factor, packed the same way
HQS_DEV float2 cfma_r(float2 a, float s, float2 acc) {
    float2 r;
    asm("{\n\t.reg .b64 p, q, t, u;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %4};\n\tmov.b64 t, {%5, %6};\n\t"
        "fma.rn.f32x2 u, p, q, t;\n\tmov.b64 {%0, %1}, u;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(s), "f"(acc.x), "f"(acc.y));
    return r;
}
HQS_DEV float2 cmul_r(float2 a, float s) {
    float2 r;
    asm("{\n\t.reg .b64 p, q, u;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %4};\n\t"
        "mul.rn.f32x2 u, p, q;\n\tmov.b64 {%0, %1}, u;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(s));
    return r;
}
// acc + a b component by component (a real factor kept as a pair)
HQS_DEV float2 cfma2(float2 a, float2 b, float2 acc) {
    float2 r;
    asm("{\n\t.reg .b64 p, q, t, u;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tmov.b64 t, {%6, %7};\n\t"
        "fma.rn.f32x2 u, p, q, t;\n\tmov.b64 {%0, %1}, u;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(acc.x), "f"(acc.y));
    return r;
}
HQS_DEV float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
HQS_DEV float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
HQS_DEV float2 cmulc(float2 a, float2 b) {
    return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
HQS_DEV float2 cfma(float2 a, float2 b, float2 acc) {   // acc + a*b
    acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
    return acc;
}
// 16-byte asynchronous copy global -> shared through L2 (cp.async.cg; both
// addresses 16-byte aligned), and the wait for every copy this thread issued.
HQS_DEV void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
// 8-byte form (through L1; both addresses 8-byte aligned)
HQS_DEV void cp_async8(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gmem_src) : "memory");
}
HQS_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> HQS_DEV void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
HQS_DEV void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch (kernels launched with launch_pdl): the
// kernel lets the next kernel of the stream launch its CTAs early and waits
// until the previous kernel of the stream has completed and its memory is
// visible; both are no-ops without a programmatic dependency.  A kernel entered
// this way touches no global memory before the wait.
HQS_DEV void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
HQS_DEV void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#define HQS_PDL_ENTRY()              \
    do {                             \
        griddep_launch_dependents(); \
        griddep_wait();              \
    } while (0)

// multiply by -i (forward) or +i (inverse)
template <bool INV> HQS_DEV float2 mul_mi(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// ---------------------------------------------------------------- errors
#define HQS_CUDA_TRY(expr)                                   \
    do {                                                     \
        cudaError_t e_ = (expr);                             \
        if (e_ != cudaSuccess) {                             \
            hqs_note_cuda_error(e_, #expr, __FILE__, __LINE__); \
            return (e_ == cudaErrorMemoryAllocation) ? HQS_ERR_OOM : HQS_ERR_CUDA; \
        }                                                    \
    } while (0)

// Keeps the message for hqs_status_string and clears the runtime's own record of the
// error: left there, an allocation that failed would be taken for the failure of the next
// launch that is checked.
void hqs_note_cuda_error(cudaError_t e, const char* what, const char* file, int line);
template <class T> static inline cudaError_t hqs_malloc(T** p, size_t bytes) {
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), bytes);
    if (e != cudaSuccess) hqs_note_cuda_error(e, "cudaMalloc", __FILE__, __LINE__);
    return e;
}

// Device error word bits (per plan), read back at sync points.
#define HQS_DEVERR_TIMEOUT   1u

// Launch with programmatic stream serialisation: the kernel's CTAs may start
// while the previous kernel of the stream finishes (the kernel begins with
// HQS_PDL_ENTRY), which hides the launch gap between the passes of an operator.
template <class... KArgs, class... Args>
static inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                     Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// ---------------------------------------------------------------- math
static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
static inline int64_t ceil_div64(int64_t a, int64_t b) { return (a + b - 1) / b; }
