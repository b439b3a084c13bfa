// Shared host/device helpers of libtiga (CUDA side only; the CPU oracle shares nothing with this).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include "tiga.h"

namespace tiga {

#define TIGA_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) return TIGA_ERR_CUDA;          \
    } while (0)

// Peek (do not clear sticky errors of other users of the context) after a launch.
static inline tiga_status launch_status() {
    return cudaPeekAtLastError() == cudaSuccess ? TIGA_OK : TIGA_ERR_CUDA;
}

// Every kernel launch of the library goes through counted(): the grid size passes through unchanged
// and the process-wide launch counter (read by tiga_kernel_launches) goes up by one.
void note_launch();
template <typename T>
static inline T counted(T grid) { note_launch(); return grid; }

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// A bump allocator over the caller's workspace (256-byte granules).
struct Carver {
    char* base;
    size_t off;
    explicit Carver(void* p) : base(static_cast<char*>(p)), off(0) {}
    template <typename T>
    T* take(size_t count) {
        T* r = reinterpret_cast<T*>(base + off);
        off += align_up(count * sizeof(T), 256);
        return r;
    }
};

// Checked build (-DTIGA_CHECKED, libtiga_checked.so): every index that is about to address a gathered row,
// an edge or a point is range-checked first; a violation sets a bit of a status word (one word per
// translation unit, read through tiga_checked_status) and the access goes to element 0 instead.  Nothing
// traps, so the context stays usable.  In the normal build checked() is the identity.
enum : unsigned { CHECK_SOURCE = 1u, CHECK_EDGE = 2u, CHECK_POINT = 4u, CHECK_SLOT = 8u };
#ifdef TIGA_CHECKED
static __device__ unsigned int g_check_status;
template <typename I>
__device__ __forceinline__ I checked(I idx, long long n, unsigned code) {
    if ((long long)idx < 0 || (long long)idx >= n) { atomicOr(&g_check_status, code); return I(0); }
    return idx;
}
// whether [first, first + len) lies within n entries; a range that does not is for the caller to read entry by entry, through checked()
__device__ __forceinline__ bool checked_range(int first, int len, long long n, unsigned code) {
    const bool whole = len <= 0 || (first >= 0 && (long long)first + len <= n);
    if (!whole) atomicOr(&g_check_status, code);
    return whole;
}
static inline unsigned read_check_status(bool reset) {
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_check_status, sizeof(v)) != cudaSuccess) return 0x80000000u;
    if (reset) cudaMemcpyToSymbol(g_check_status, &z, sizeof(z));
    return v;
}
#else
template <typename I>
__device__ __forceinline__ I checked(I idx, long long, unsigned) { return idx; }
__device__ __forceinline__ bool checked_range(int, int, long long, unsigned) { return true; }
static inline unsigned read_check_status(bool) { return 0u; }
#endif
// one reader per translation unit (defined at the end of every .cu file), combined by tiga_checked_status
unsigned check_status_csr(bool reset);
unsigned check_status_csr_plan(bool reset);
unsigned check_status_csr_attention(bool reset);
unsigned check_status_radius(bool reset);
unsigned check_status_radius_lj(bool reset);
unsigned check_status_radius_mlp(bool reset);
unsigned check_status_knn(bool reset);

// two fp32 values per register pair: sm_100 executes add / mul / fma on both with one instruction
typedef unsigned long long f32x2;
static __device__ __forceinline__ f32x2 pack2(float a, float b) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
static __device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
static __device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { f32x2 r; asm("sub.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
static __device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { f32x2 r; asm("add.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
static __device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { f32x2 r; asm("mul.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
static __device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
static __device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }

// streaming (read-once) loads and write-once stores keep L2 for the gathered rows
template <typename T>
__device__ __forceinline__ T ld_stream(const T* p) { return __ldcs(p); }
template <typename T>
__device__ __forceinline__ void st_stream(T* p, T v) { __stcs(p, v); }

}  // namespace tiga
