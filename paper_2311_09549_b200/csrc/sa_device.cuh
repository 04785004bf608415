// Small device helpers shared by the kernels.
#pragma once

#include <cuda_runtime.h>
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "sa_internal.h"

#define SA_FULL_MASK 0xffffffffu

// fp32 numbers that an earlier kernel on the stream may have written: dense operands, temporaries, partial sums.  A kernel may
// start while that one is still running (sa_launch), so they are not constant for its lifetime, which is what __ldg,
// ld.global.nc and `const float *__restrict__` promise: the compiler may move such loads up across the wait, and the read-only
// path need not see the new values.  A kernel takes them as sa_input; what sa_after_previous returns turns that into sa_data,
// whose loads are coherent and take the number that the wait gave as an operand (unused, no instruction), so that they stay
// behind it and are otherwise free to move: with all of them volatile, their order fixed, kernel 1 on 60 K nonzeros
// in long rows (K = L = 128) took 24.1 us instead of 20.5.  (The _here loads are volatile where a loop's loads are placed by
// hand: the rows in flight of the order-3 kernel and the dense stage, and kernel 8's rows of C, which spill when left free.)
// Work lists and the tensor's arrays (sa_values: its values) are never written by a kernel; they take the read-only path.
struct sa_input {
    const float *p;
    __host__ __device__ __forceinline__ sa_input(const float *q) : p(q) {}
};
struct sa_values {
    const float *p;
    __host__ __device__ __forceinline__ sa_values(const float *q) : p(q) {}
};
struct sa_ready;
class sa_data {
    uint32_t ready;
    __device__ __forceinline__ sa_data(const float *q, uint32_t r) : ready(r), p(q) {}
    friend struct sa_ready;

public:
    const float *p;
    __device__ __forceinline__ sa_data operator+(int64_t n) const { return sa_data(p + n, ready); }
    __device__ __forceinline__ sa_data plus_bytes(uint64_t n) const
    {
        return sa_data(reinterpret_cast<const float *>(reinterpret_cast<const char *>(p) + n), ready);
    }
    __device__ __forceinline__ float ld() const
    {
        float v;
        asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p), "r"(ready));
        return v;
    }
    __device__ __forceinline__ float ld_cs() const             // read once: evict first
    {
        float v;
        asm("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p), "r"(ready));
        return v;
    }
    __device__ __forceinline__ float2 ld2() const
    {
        float2 v;
        asm("ld.global.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p), "r"(ready));
        return v;
    }
    __device__ __forceinline__ float4 ld4() const
    {
        float4 v;
        asm("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "r"(ready));
        return v;
    }
    __device__ __forceinline__ float4 ld4_cs() const
    {
        float4 v;
        asm("ld.global.cs.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "r"(ready));
        return v;
    }
    __device__ __forceinline__ float4 ld4_once() const         // not kept in L1
    {
        float4 v;
        asm("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "r"(ready));
        return v;
    }
    // the same in its place among the other volatile statements
    __device__ __forceinline__ float2 ld2_here() const
    {
        float2 v;
        asm volatile("ld.global.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
        return v;
    }
    __device__ __forceinline__ float4 ld4_here() const
    {
        float4 v;
        asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
        return v;
    }
    __device__ __forceinline__ float4 ld4_once_here() const
    {
        float4 v;
        asm volatile("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
        return v;
    }
};
struct sa_ready {
    uint32_t token;
    __device__ __forceinline__ sa_data operator()(sa_input in) const { return sa_data(in.p, token); }
};

// Streaming (evict-first) stores for output tiles that are written once and never re-read, so
// they do not displace the factor matrices held in L2.
__device__ __forceinline__ void sa_st_cs(float *p, float v) { __stcs(p, v); }
__device__ __forceinline__ void sa_st_cs4(float *p, float4 v) { __stcs(reinterpret_cast<float4 *>(p), v); }
__device__ __forceinline__ void sa_st_cs2(float *p, float2 v) { __stcs(reinterpret_cast<float2 *>(p), v); }

// Self-checking build (-DSA_DEBUG_BOUNDS): every index that comes out of the tensor's arrays is checked before it
// is turned into an address; the first violation is recorded in the tensor's status word (check number, offending
// value, thread; read back by sa_last_device_status / sa_device_status_words) and the caller redirects the access to
// a valid element.  Nothing traps.  In the normal build SA_CHK is the constant true.
#ifdef SA_DEBUG_BOUNDS
__device__ __forceinline__ bool sa_dbg_ok(int32_t *status, bool ok, int code, int64_t value)
{
    if (!ok && atomicCAS(status, 0, int(SA_E_BOUNDS)) == 0) {
        status[1] = code;
        status[2] = int32_t(value);
        status[3] = int32_t(blockIdx.x * blockDim.x + threadIdx.x);
    }
    return ok;
}
#define SA_CHK(status, cond, code, value) sa_dbg_ok(status, cond, code, int64_t(value))
#else
#define SA_CHK(status, cond, code, value) true
#endif

// What the checks of the row / fiber kernels compare against: rows of the gathered dense operand(s), output rows,
// partial slots, nonzeros (items come from the work lists, indices from crd).
struct sa_limits {
    int32_t *status;
    uint32_t gather_rows, out_rows;
    int32_t n_slots, nnz;
};

static inline sa_limits sa_make_limits(const sa_tensor *t, int64_t gather_rows, int64_t out_rows, int64_t n_slots)
{
    sa_limits lim;
    lim.status = t->d_status;
    lim.gather_rows = uint32_t(gather_rows);
    lim.out_rows = uint32_t(out_rows);
    lim.n_slots = int32_t(n_slots);
    lim.nnz = int32_t(t->nnz);
    return lim;
}

// Programmatic dependent launch: a kernel's blocks come onto the SMs when the last block of the kernel before it has left, read
// there what no kernel ever writes (work lists, the tensor's arrays) and wait, in sa_after_previous, until that kernel is through
// and its results can be seen.  Nothing else may be read or written before that, and some thread of every launch has to wait,
// or a kernel further back could still be running.
// No kernel lets the next one start before its own blocks have left (griddepcontrol.launch_dependents): the next one's blocks
// then came onto the SMs as these emptied, several onto the first ones, and ran to their end with the split of L1 and shared
// memory that they found there.  Two calls in turn, us, ordinary launches / with launch_dependents behind the wait (and only
// kernels of a block per SM, or with no need of L1, starting early) / as it is: row kernel on 60 K nonzeros and kernel 1 on
// 100 K (K = L = 128) 55 / 87 / 51, order 3 on 8 M nonzeros and the same kernel 1 176 / 194 / 169.  One call after another:
// kernel 1 on 6 M nonzeros 234 / 236 / 233, kernel 2 on 60 K (three launches) 18.4 / 13.8 / 12.3, kernel 7 on 60 K 12.6 / 11.9 /
// 7.0, order 3 on 20 K (one launch, the one that is slower so) 10.3 / 7.7 / 8.1.
__device__ __forceinline__ sa_ready sa_after_previous()
{
    sa_ready r;
    asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(r.token) : : "memory");
    return r;
}

// The arguments convert as they do in a call (not by a cast: a pointer in the wrong place does not compile).
template <typename T>
struct sa_arg { using type = T; };
template <typename... Params>
static inline cudaError_t sa_launch(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream,
                                    typename sa_arg<Params>::type... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    static_assert(!(std::is_same<Params, const float *>::value || ...), "fp32 inputs are sa_input or sa_values");
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Opt a kernel into `bytes` of dynamic shared memory once per device instead of once per launch (the attribute is
// per device; `done` is the caller's flags, one per device ordinal).  Host threads may launch at the same time: the
// attribute may then be set more than once, to the same value.
constexpr int SA_MAX_DEVICE_FLAGS = 64;
struct sa_device_flags { std::atomic<bool> set[SA_MAX_DEVICE_FLAGS]; };
template <typename Kernel>
static inline bool sa_set_smem_once(Kernel kernel, int bytes, sa_device_flags &done)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const bool keep = dev >= 0 && dev < SA_MAX_DEVICE_FLAGS;
    if (keep && done.set[dev].load(std::memory_order_acquire)) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (keep) done.set[dev].store(true, std::memory_order_release);
    return true;
}

// ---- PTX helpers shared by the kernels

// x = hi + lo + rest in TF32 numbers: hi the upper 19 bits of x, lo the upper 19 bits of x - hi (exact in fp32).  hi.hi +
// hi.lo + lo.hi then misses the true product by about 2^-20 relative.  (cvt.rna.tf32 costs several instructions per value on
// this target; plain masking is one.)
__device__ __forceinline__ void split_tf32(float x, uint32_t &hi, uint32_t &lo)
{
    hi = __float_as_uint(x) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi)) & 0xffffe000u;
}

__device__ __forceinline__ void mma_m16n8k8_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void cp_async16_raw(uint32_t dst_smem, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Sum `count` partial tiles into out rows (count == 0: zero fill).  A tile is 2^shift float4, shift > 5.  The builder puts the
// entries with the most partials first.  Blocks of 256 threads, W float4 columns x 256 / W phases over the partials: W = 16
// for the first n_big entries (more than SA_BIG_FIX partials), 64 up to entry n_sum, tile / W blocks each; the entries behind
// are zeroed 256 float4 per block.  Fixed summation order: deterministic.  192 partials of 4 KB: 13 us with 64 columns per
// block throughout, 7.5 us.
static __global__ void __launch_bounds__(256)
sa_fixup_kernel(const sa_fix *__restrict__ fix, unsigned n_big, unsigned n_sum, unsigned n_fix, sa_input partial_in,
                float *__restrict__ out, int shift)
{
    __shared__ float4 red[256];
    const sa_data partial = sa_after_previous()(partial_in);
    const unsigned big_blocks = n_big << (shift - 4), sum_blocks = (n_sum - n_big) << (shift - 6);
    unsigned b = blockIdx.x;
    if (b >= big_blocks + sum_blocks) {
        const int64_t z = int64_t(b - big_blocks - sum_blocks) * 256 + threadIdx.x, e = n_sum + (z >> shift);
        if (e < n_fix)
            sa_st_cs4(out + ((int64_t(fix[e].out_row) << shift) + (z & ((1 << shift) - 1))) * 4, make_float4(0.f, 0.f, 0.f, 0.f));
        return;
    }
    const bool big = b < big_blocks;
    if (!big) b -= big_blocks;
    const int wlog = big ? 4 : 6, W = 1 << wlog, P = 256 >> wlog;
    const sa_fix e = fix[(big ? 0 : n_big) + (b >> (shift - wlog))];
    const int col = threadIdx.x & (W - 1), phase = threadIdx.x >> wlog;
    const int64_t f4 = int64_t(b & ((1u << (shift - wlog)) - 1)) * W + col;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const sa_data base = partial + ((int64_t(e.slot0) << shift) + f4) * 4;
#pragma unroll 4
    for (int q = phase; q < e.count; q += P) {
        const float4 v = (base + ((int64_t(q) << shift) * 4)).ld4();
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (phase == 0) {
        for (int q = 1; q < P; ++q) {
            const float4 v = red[q * W + col];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        sa_st_cs4(out + ((int64_t(e.out_row) << shift) + f4) * 4, s);
    }
}

// The same for rows of at most 128 floats (8, 16 or 32 float4): the first n_big entries (the builder puts the longest
// first) take a block each as above, the others a warp each, which is all that a few partial rows can use.
static __global__ void __launch_bounds__(256)
sa_fixup_rows_kernel(const sa_fix *__restrict__ fix, int n_fix, int n_big, sa_input partial_in, float *__restrict__ out,
                     int row_floats)
{
    __shared__ float4 red[256];
    const bool big = int(blockIdx.x) < n_big;
    const int W = row_floats / 4, lane = threadIdx.x & 31;
    const int entry = big ? int(blockIdx.x) : n_big + (int(blockIdx.x) - n_big) * 8 + int(threadIdx.x >> 5);
    if (entry >= n_fix) return;                        // whole warps of the last block
    const sa_fix e = fix[entry];
    const sa_data partial = sa_after_previous()(partial_in);
    const int who = big ? int(threadIdx.x) : lane, P = (big ? 256 : 32) / W;
    const int col = who % W, phase = who / W;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const sa_data base = partial + (int64_t(e.slot0) * row_floats + col * 4);
#pragma unroll 4
    for (int q = phase; q < e.count; q += P) {
        const float4 v = (base + int64_t(q) * row_floats).ld4();
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    red[threadIdx.x] = s;
    if (big) __syncthreads();
    else __syncwarp();
    if (phase == 0) {
        const float4 *mine = red + (big ? 0 : int(threadIdx.x) - lane);
        for (int q = 1; q < P; ++q) {
            const float4 v = mine[q * W + col];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        sa_st_cs4(out + int64_t(e.out_row) * row_floats + col * 4, s);
    }
}

static inline cudaError_t sa_launch_fixup(const sa_worklist &wl, const float *partial, float *out, int tile_floats,
                                          cudaStream_t stream)
{
    if (wl.fix.empty()) return cudaSuccess;
    const int nf4 = tile_floats / 4;
    if (nf4 <= 32) {
        const unsigned rows = (unsigned)wl.fix.size(), big = (unsigned)wl.n_big_fix;
        return sa_launch(sa_fixup_rows_kernel, big + (rows - big + 7) / 8, 256, 0, stream, wl.d_fix, int(rows), int(big), partial, out,
                         tile_floats);
    }
    int shift = 0;
    while ((4 << shift) < tile_floats) ++shift;
    const int64_t zeros = int64_t(wl.fix.size()) - wl.n_sum_fix;
    const int64_t blocks = (wl.n_big_fix << (shift - 4)) + ((wl.n_sum_fix - wl.n_big_fix) << (shift - 6)) + (((zeros << shift) + 255) >> 8);
    return sa_launch(sa_fixup_kernel, unsigned(blocks), 256, 0, stream, wl.d_fix, unsigned(wl.n_big_fix), unsigned(wl.n_sum_fix),
                     unsigned(wl.fix.size()), partial, out, shift);
}
