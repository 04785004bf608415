// Kernel 1 <SDDMM,SpMM>:  A(i,l) = sum_j B(i,j) (sum_k C(i,k) D(j,k)) E(j,l), scheduled as the
// fused nest  i, j' < t ; k: t += B(i,j) C(i,k) D(j,k) , l: A(i,l) += t E(j,l) >  of the paper's
// Table of kernels (Section 6): the sampled value is a scalar temporary that is consumed at once,
// the sampled matrix is never written (auxiliary memory 1 in the paper's memory table; what the workspace holds are partial
// rows of long rows: L floats per 32 nonzeros at most, per 16 where the matrix is small).
//
// A warp is four groups of eight lanes; every group takes one work item (a range of short rows, or a piece of a long
// row) and walks its nonzeros U at a time: a lane owns the float4 columns l, l + 8, ... of D(j,:), E(j,:), C(i,:) and of
// the output row, so a row piece of 128 bytes is one load instruction of the group, a dot product is three shuffles per
// four nonzeros of the warp, and nothing passes through shared memory.  Indices and values come as 8-byte records that
// all lanes of a group read (one step ahead); C(i + 1,:) is requested while row i is being summed.
// What bounds it: the gathered rows of D and E.  Where they exceed L2 the builder cuts long rows at column-block
// boundaries and orders the pieces by block (build_sddmm), so that what runs at one time gathers from a few blocks that
// L2 holds; what then limits is the L2-to-SM path (4 (K + L) bytes per nonzero), not HBM.  1M x 1M, 30 M nonzeros,
// K = L = 64: 1.01 ms, 15.7 GB through that path and 2.8 GB of DRAM traffic, where one warp per item with the rows in a
// cp.async ring and items in order of size took 2.24 ms and 13.2 GB.  Two nonzeros per step with 24 warps per SM: 9 % slower.
#include "sa_device.cuh"

namespace {

template <int K, int L>
struct sd_cfg {
    static constexpr int DQ = K / 32, EQ = L / 32;    // float4 pieces of D(j,:) and E(j,:) per lane
    static constexpr int U = DQ + EQ <= 4 ? 4 : 2;    // nonzeros per group and step: 16 float4 in flight per lane at most
    static constexpr bool AHEAD = DQ + EQ < 8;        // C of the next row in registers (spills at K = L = 128)
    // Blocks per SM.  K = L = 32 has half the bytes in flight per lane and needs the warps: 100 K rows of 100 nonzeros on 1 M
    // columns 337 us with two blocks, 273 with three, 489 (spills) with four; eight nonzeros per step with two blocks 307.
    static constexpr int CTAS = DQ + EQ <= 2 ? 3 : 2;
};

template <int K, int L, int CTAS>
__global__ void __launch_bounds__(256, CTAS)
sddmm_spmm_kernel(const sa_item *__restrict__ items, int64_t n_items, const int32_t *__restrict__ pos,
                  const int2 *__restrict__ nz, sa_input C_in, uint32_t ldc, sa_input D_in, uint32_t ldd, sa_input E_in, uint32_t lde,
                  float *__restrict__ out, float *__restrict__ partial, float *__restrict__ sampled, const sa_limits lim)
{
    using G = sd_cfg<K, L>;
    constexpr int DQ = G::DQ, EQ = G::EQ, U = G::U;
    const int l = threadIdx.x & 7;
    const int64_t idx = (int64_t(blockIdx.x) * 256 + threadIdx.x) >> 3;
    int r = 0, rend = 0, p = 0, end = 0, dest = -1;
    if (idx < n_items) {
        const int4 ia = __ldg(reinterpret_cast<const int4 *>(items + idx));          // out_row, row_end, -, -
        const int4 ib = __ldg(reinterpret_cast<const int4 *>(items + idx) + 1);      // p0, p1, dest, -
        if (SA_CHK(lim.status, ia.x >= 0 && ia.x <= ia.y && uint32_t(ia.y) <= lim.out_rows && ib.x >= 0 && ib.x <= ib.y && ib.y <= lim.nnz &&
                                   ib.z < lim.n_slots, 43, idx)) {
            r = ia.x; rend = ia.y; p = ib.x; end = ib.y; dest = ib.z;
        }
    }
    // [p, b): what is left of row r; bn: where row r + 1 ends; c, cn: C of both rows
    float4 c[DQ], cn[DQ], acc[EQ];
    auto row_end = [&](int row) {
        if (dest >= 0 || row >= rend) return end;
        int e = __ldg(pos + row + 1);
        if (!SA_CHK(lim.status, e >= 0 && e <= end, 44, e)) e = end;
        return e;
    };
    int b = row_end(r), bn = row_end(r + 1);
    int2 rec[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        rec[u] = make_int2(0, 0);
        if (p + u < end) rec[u] = __ldg(nz + p + u);
    }
    const sa_ready ready = sa_after_previous();
    const sa_data C = ready(C_in), Dl = ready(D_in) + 4 * l, El = ready(E_in) + 4 * l;
    auto load_c = [&](float4 (&x)[DQ], int row) {
        if (row < rend) {
#pragma unroll
            for (int q = 0; q < DQ; ++q) x[q] = (C + (uint32_t(row) * ldc + 32u * q + 4u * l)).ld4();
        }
    };
    load_c(c, r);
    if (G::AHEAD) load_c(cn, r + 1);
#pragma unroll
    for (int q = 0; q < EQ; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t d_bytes = ldd * 4u, e_bytes = lde * 4u;
    for (;;) {
        while (p == b && r < rend) {                  // the row is complete (or empty: +0)
            float *dst = (dest >= 0 ? partial + int64_t(dest) * L : out + int64_t(r) * L) + 4 * l;
#pragma unroll
            for (int q = 0; q < EQ; ++q) {
                *reinterpret_cast<float4 *>(dst + 32 * q) = acc[q];
                acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            ++r;
            b = bn;
            bn = row_end(r + 1);
            if (G::AHEAD) {
#pragma unroll
                for (int q = 0; q < DQ; ++q) c[q] = cn[q];
                load_c(cn, r + 1);
            } else {
                load_c(c, r);
            }
        }
        if (!__any_sync(SA_FULL_MASK, r < rend)) break;
        const int n = min(U, b - p);                  // 0 for a group that is done
        float4 d[U][DQ], e[U][EQ];
        float v[U], dot[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            dot[u] = 0.f;
            v[u] = __int_as_float(rec[u].y);
            if (u < n) {
                uint32_t j = uint32_t(rec[u].x);
                if (!SA_CHK(lim.status, j < lim.gather_rows, 42, j)) j = 0u;
#pragma unroll
                for (int q = 0; q < DQ; ++q) d[u][q] = (Dl.plus_bytes(uint64_t(j) * d_bytes) + 32 * q).ld4();
#pragma unroll
                for (int q = 0; q < EQ; ++q) e[u][q] = (El.plus_bytes(uint64_t(j) * e_bytes) + 32 * q).ld4();
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)                   // the next step's records (rows of a range lie one after the other)
            if (p + n + u < end) rec[u] = __ldg(nz + p + n + u);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u < n) {
#pragma unroll
                for (int q = 0; q < DQ; ++q)
                    dot[u] = fmaf(c[q].x, d[u][q].x, fmaf(c[q].y, d[u][q].y, fmaf(c[q].z, d[u][q].z, fmaf(c[q].w, d[u][q].w, dot[u]))));
            }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < U; ++u) dot[u] += __shfl_xor_sync(SA_FULL_MASK, dot[u], o);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u < n) {
                const float sc = v[u] * dot[u];
                if (sampled != nullptr && l == 0) sampled[p + u] = sc;
#pragma unroll
                for (int q = 0; q < EQ; ++q) {
                    acc[q].x = fmaf(sc, e[u][q].x, acc[q].x);
                    acc[q].y = fmaf(sc, e[u][q].y, acc[q].y);
                    acc[q].z = fmaf(sc, e[u][q].z, acc[q].z);
                    acc[q].w = fmaf(sc, e[u][q].w, acc[q].w);
                }
            }
        p += n;
    }
}

template <int K, int L>
cudaError_t launch(const sa_tensor *t, const sa_dense *ops, float *out, float *partial, float *sampled,
                   cudaStream_t stream)
{
    const sa_worklist &wl = t->wl_main;
    const int64_t n_items = int64_t(wl.items.size());
    const int64_t ctas = (n_items + 31) / 32;         // 32 groups per block
    if (ctas == 0) return cudaSuccess;
    // Up to three rounds of items the length of one is the run time, and two blocks per SM walk it faster (registers for
    // more loads at a time).  K = L = 32, us, two / three blocks: 60 K nonzeros (4.7 K items) 14.4 / 16.5, 1 M on 20 K rows
    // (22 K items) 29.3 / 31.8, 400 K on 40 K rows (26 K) 29.1 / 30.9, 1.5 M on 50 K rows (30 K) 48.3 / 47.5, 1 M on 300 K rows
    // (38 K) 61 / 53, on 200 K rows and 700 K columns (42 K) 83 / 69.
    auto kern = n_items <= int64_t(3) * 2 * SA_SMS * 32 ? sddmm_spmm_kernel<K, L, 2> : sddmm_spmm_kernel<K, L, sd_cfg<K, L>::CTAS>;
    sa_launch(kern, (unsigned)ctas, 256, 0, stream, wl.d_items, n_items, t->d_pos[1], t->d_nzpack, ops[0].ptr, uint32_t(ops[0].ld),
              ops[1].ptr, uint32_t(ops[1].ld), ops[2].ptr, uint32_t(ops[2].ld), out, partial, sampled,
              sa_make_limits(t, t->dims[1], t->dims[0], wl.n_slots));
    return cudaGetLastError();
}

bool rank_ok(int64_t r) { return r == 32 || r == 64 || r == 128; }

}  // namespace

bool sa_ranks_ok_sddmm(int64_t K, int64_t L) { return rank_ok(K) && rank_ok(L); }

// workspace: [partial rows of long-row pieces][sampled values, nnz floats, debug schedule only]
size_t sa_ws_sddmm_spmm(const sa_tensor *t, const sa_dense *ops, bool materialize)
{
    size_t b = sa_align256(size_t(t->wl_main.n_slots) * size_t(ops[2].cols) * sizeof(float));
    if (materialize) b += sa_align256(size_t(t->nnz) * sizeof(float));
    return b;
}

sa_status sa_launch_sddmm_spmm(const sa_tensor *t, const sa_dense *ops, float *out, void *ws, size_t, bool materialize,
                               cudaStream_t stream, int *launches)
{
    const int64_t K = ops[0].cols, L = ops[2].cols;
    float *partial = static_cast<float *>(ws);
    float *sampled = nullptr;
    for (int i = 0; i < 3; ++i)                       // rows of C are found by 32-bit offsets; one limit for all operands
        if (ops[i].rows * ops[i].ld >= (int64_t(1) << 30)) return SA_E_UNSUPPORTED;
    if (materialize)
        sampled = reinterpret_cast<float *>(static_cast<char *>(ws) + sa_align256(size_t(t->wl_main.n_slots) * size_t(L) * sizeof(float)));
    cudaError_t e = cudaErrorInvalidValue;
#define SA_CASE(a, b) if (K == a && L == b) e = launch<a, b>(t, ops, out, partial, sampled, stream);
    SA_CASE(32, 32) SA_CASE(32, 64) SA_CASE(32, 128) SA_CASE(64, 32) SA_CASE(64, 64) SA_CASE(64, 128)
    SA_CASE(128, 32) SA_CASE(128, 64) SA_CASE(128, 128)
#undef SA_CASE
    if (e != cudaSuccess) return SA_E_CUDA;
    *launches = t->wl_main.items.empty() ? 0 : 1;
    if (!t->wl_main.fix.empty()) {
        if (sa_launch_fixup(t->wl_main, partial, out, int(L), stream) != cudaSuccess) return SA_E_CUDA;
        *launches += 1;
    }
    return SA_OK;
}

// ---- kernel 2 <SDDMM,SpMM,GEMM>:  A(i,m) = sum_{j,k,l} B(i,j) C(i,k) D(j,k) E(j,l) F(l,m), the two-level
// schedule  i < T(l) ; j' < t ; k: ... , l: T(l) += t E(j,l) > , m,l: A(i,m) += T(l) F(l,m) >  of the paper's
// Table of kernels: the row temporary T is what the fused kernel above produces per row; here it goes
// through the workspace (I x L floats) to a tensor-core product with F instead of staying in registers.
// workspace: [T: I x L][partial rows of long-row pieces]
size_t sa_ws_sddmm_spmm_gemm(const sa_tensor *t, const sa_dense *ops)
{
    return sa_align256(size_t(t->dims[0]) * size_t(ops[2].cols) * sizeof(float)) + sa_ws_sddmm_spmm(t, ops, false);
}

sa_status sa_launch_sddmm_spmm_gemm(const sa_tensor *t, const sa_dense *ops, float *out, void *ws, size_t ws_bytes,
                                    cudaStream_t stream, int *launches)
{
    const int64_t I = t->dims[0], L = ops[2].cols, M = ops[3].cols;
    const size_t t_bytes = sa_align256(size_t(I) * size_t(L) * sizeof(float));
    float *T = static_cast<float *>(ws);
    int n1 = 0;
    const sa_status s = sa_launch_sddmm_spmm(t, ops, T, static_cast<char *>(ws) + t_bytes, ws_bytes - t_bytes, false, stream, &n1);
    if (s != SA_OK) return s;
    const sa_status g = sa_launch_dense_gemm(I, T, L, ops[3].ptr, ops[3].ld, L, M, out, t->d_status, stream);
    if (g != SA_OK) return g;
    *launches = n1 + 1;
    return SA_OK;
}
