// Kernel 5 <3D TTMC>:  A(l,m,n) = sum_{i,j,k} B(i,j,k) C(i,l) D(j,m) E(k,n)  (the running example of
// the paper, Sections 1 and 3; chosen schedules in the Table of kernels, Section 6).  Evaluated as
//   T(i,m,n) = sum_j D(j,m) ( sum_k B(i,j,k) E(k,n) )        per slice, the branched nest of kernel 6
//   A(l,m,n) = sum_i C(i,l) T(i,m,n)                         contraction over the slices
// in two schedules:
//   SA_SCHED_FUSED      the paper's second schedule for this kernel with its temporaries widened to
//     vectors: i < T(m,n) ; j' < t(n) ; k': t += B E , m: T += t D > , l: A += T C >.  The slice
//     temporary stays on chip; every thread block keeps its own L x M x N accumulator in shared
//     memory (sa_ttm3.cu, ttmc3_fused_kernel) and the blocks' accumulators are added in block order.
//     Additions inside a block are shared-memory atomics: their order, and with it the last bits of
//     the result, may differ from run to run.
//   SA_SCHED_FISSIONED  the loop over i is fissioned from the l loop: the slice temporaries T(i,:,:)
//     (I x M x N floats, in the workspace) are written by the slice kernel of kernel 6 and reduced
//     over i by a small dense kernel (fixed chunks of slices, partial sums added in a fixed order:
//     bitwise reproducible).  A temporary of three dimensions is what Stage 1 of the paper's
//     auto-scheduler prunes; it is kept as the reproducible alternative and for rank combinations
//     whose accumulator does not fit shared memory.
#include <algorithm>

#include "sa_device.cuh"

namespace {

constexpr int TTMC_MAX_CHUNKS = 512;

// P(c, l, col) = sum over the slices i of chunk c of C(i,l) * T(i,col).  One thread per column, C(i,:) of TTMC_STEP slices in
// shared memory, eight rows of T requested at a time: with one row at a time the chain of loads was the run time (12 K slices,
// L = 16, 256 columns: 36 us, now 13 us).
constexpr int TTMC_STEP = 64;
template <int L>
__global__ void __launch_bounds__(256)
ttmc3_partial_kernel(int64_t I, int chunk, int cols, sa_input T_in, sa_input C_in, uint32_t ldc, float *__restrict__ P)
{
    __shared__ __align__(16) float cs[TTMC_STEP * L];
    const sa_ready ready = sa_after_previous();
    const sa_data T = ready(T_in), C = ready(C_in);
    const int col = blockIdx.x * 256 + threadIdx.x;
    const int64_t i0 = int64_t(blockIdx.y) * chunk, i1 = min(I, i0 + chunk);
    float acc[L];
#pragma unroll
    for (int l = 0; l < L; ++l) acc[l] = 0.f;
    for (int64_t base = i0; base < i1; base += TTMC_STEP) {
        const int n = int(min(int64_t(TTMC_STEP), i1 - base));
        __syncthreads();
        for (int x = threadIdx.x * 4; x < n * L; x += 1024)
            *reinterpret_cast<float4 *>(cs + x) = (C + ((base + x / L) * ldc + x % L)).ld4();
        __syncthreads();
        const sa_data t0 = T + (base * cols + col);
        for (int s = 0; s < n; s += 8) {
            float t[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) t[u] = s + u < n ? (t0 + int64_t(s + u) * cols).ld_cs() : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (s + u >= n) break;
                const float *c = cs + (s + u) * L;
#pragma unroll
                for (int l = 0; l < L; l += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(c + l);
                    acc[l + 0] = fmaf(w.x, t[u], acc[l + 0]);
                    acc[l + 1] = fmaf(w.y, t[u], acc[l + 1]);
                    acc[l + 2] = fmaf(w.z, t[u], acc[l + 2]);
                    acc[l + 3] = fmaf(w.w, t[u], acc[l + 3]);
                }
            }
        }
    }
    float *dst = P + (int64_t(blockIdx.y) * L) * cols + col;
#pragma unroll
    for (int l = 0; l < L; ++l) dst[int64_t(l) * cols] = acc[l];
}

// A(x) = sum over chunks c of P(c, x), x = l * cols + col, in a fixed order: 16 phases over the chunks (64 outputs per block),
// then the phases.  188 chunks of 4096: 17 us as one sum per thread, 8 us now.
__global__ void __launch_bounds__(256)
ttmc3_final_kernel(int n_chunks, int64_t n_out, sa_input P_in, float *__restrict__ A)
{
    __shared__ float4 red[256];
    const sa_data P = sa_after_previous()(P_in);
    const int col = threadIdx.x & 15, phase = threadIdx.x >> 4;
    const int64_t x = (int64_t(blockIdx.x) * 16 + col) * 4;               // n_out is a multiple of 64
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int c = phase; c < n_chunks; c += 16) {
        const float4 v = (P + (int64_t(c) * n_out + x)).ld4();
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (phase == 0) {
        for (int q = 1; q < 16; ++q) {
            const float4 v = red[q * 16 + col];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4 *>(A + x) = s;
    }
}

struct ttmc3_plan {
    int chunk, n_chunks;
    size_t t_bytes, ttm3_bytes, p_bytes;
};

ttmc3_plan plan(const sa_tensor *t, const sa_dense *ops)
{
    ttmc3_plan p;
    const int64_t I = t->dims[0], L = ops[0].cols, cols = ops[1].cols * ops[2].cols;
    p.chunk = int(std::max<int64_t>(64, (I + TTMC_MAX_CHUNKS - 1) / TTMC_MAX_CHUNKS));
    p.n_chunks = int((I + p.chunk - 1) / p.chunk);
    p.t_bytes = sa_align256(size_t(I) * size_t(cols) * sizeof(float));
    p.ttm3_bytes = sa_ws_ttm3(t, ops + 1);
    p.p_bytes = sa_align256(size_t(p.n_chunks) * size_t(L) * size_t(cols) * sizeof(float));
    return p;
}

}  // namespace

bool sa_ranks_ok_ttmc3(int64_t L, int64_t M, int64_t N) { return (L == 16 || L == 32) && sa_ranks_ok_ttm3(M, N); }

// workspace, fissioned: [T: I x M x N][partial tiles of the slice kernel][P: chunks x L x M x N]
//            fused:     [accumulators of the blocks: blocks x L x M x N]
size_t sa_ws_ttmc3(const sa_tensor *t, const sa_dense *ops, bool fissioned)
{
    if (!fissioned) return sa_ws_ttmc3_fused(ops[0].cols, ops[1].cols, ops[2].cols);
    const ttmc3_plan p = plan(t, ops);
    return p.t_bytes + p.ttm3_bytes + p.p_bytes;
}

sa_status sa_launch_ttmc3(const sa_tensor *t, const sa_dense *ops, float *out, void *ws, size_t, bool fissioned,
                          cudaStream_t stream, int *launches)
{
    const int64_t I = t->dims[0], L = ops[0].cols;
    const int cols = int(ops[1].cols * ops[2].cols);
    if (ops[0].rows * ops[0].ld >= (int64_t(1) << 30)) return SA_E_UNSUPPORTED;
    if (!fissioned) {
        float *partials = static_cast<float *>(ws);
        int n_blocks = 0;
        const sa_status s = sa_launch_ttmc3_fused_stage(t, ops[0], ops[1], ops[2], partials, stream, &n_blocks);
        if (s != SA_OK) return s;
        const int64_t n_out = L * cols;
        // n_blocks == 0 (a tensor without nonzeros): the sum over no accumulators writes zeros
        sa_launch(ttmc3_final_kernel, (unsigned)(n_out / 64), 256, 0, stream, n_blocks, n_out, partials, out);
        if (cudaGetLastError() != cudaSuccess) return SA_E_CUDA;
        *launches = (n_blocks > 0 ? 1 : 0) + 1;
        return SA_OK;
    }
    const ttmc3_plan p = plan(t, ops);
    char *base = static_cast<char *>(ws);
    float *T = reinterpret_cast<float *>(base);
    void *ws3 = base + p.t_bytes;
    float *P = reinterpret_cast<float *>(base + p.t_bytes + p.ttm3_bytes);
    int n3 = 0;
    const sa_status s = sa_launch_ttm3(t, ops + 1, T, ws3, p.ttm3_bytes, stream, &n3);   // T(i,m,n), empty slices zero
    if (s != SA_OK) return s;
    *launches = n3;
    dim3 grid((unsigned)(cols / 256), (unsigned)p.n_chunks);              // cols is 256, 512 or 1024
    auto kern = L == 16 ? ttmc3_partial_kernel<16> : ttmc3_partial_kernel<32>;
    sa_launch(kern, grid, 256, 0, stream, I, p.chunk, cols, T, ops[0].ptr, uint32_t(ops[0].ld), P);
    if (cudaGetLastError() != cudaSuccess) return SA_E_CUDA;
    const int64_t n_out = L * cols;
    sa_launch(ttmc3_final_kernel, (unsigned)(n_out / 64), 256, 0, stream, p.n_chunks, n_out, P, out);
    if (cudaGetLastError() != cudaSuccess) return SA_E_CUDA;
    *launches += 2;
    return SA_OK;
}
