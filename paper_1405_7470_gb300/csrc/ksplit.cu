// K-split SIMT kernel (FP32) for the element-local contraction
//     out[f,e,i] = sum_j D[f,i,j] * u[e,j]                (dG FEM volume, Table 1)
// read as the product of the u tile [BM x N] and D^T [N x F*N] (column c = f*N + i).
//
// Transformations (Section 2.4) and how they map here:
//   split_iname(e, BM)       one tile of BM elements per CTA step (persistent, grid-stride);
//                            rows past E are zeros and are not stored.
//   split_iname(j, BK)       the reduction in chunks of BK; the D^T slice of each chunk is
//                            fetched asynchronously (cp.async, 4-byte elements, zero-filled
//                            past N or past the last column) into a two-slot ring one chunk
//                            ahead, so D^T never has to fit in shared memory at once.
//   add_prefetch(u)          the u tile, transposed to [j][e], stays resident for every
//                            column block of the tile; with two buffers the next tile's
//                            u is fetched while this one is used.
//   ilp on e and on i        8 x 8 register block per thread: two quads of tile positions by
//                            two quads of column positions; the operand reads are 16-byte
//                            vector loads.
//   unr on j                 the chunk loop is fully unrolled.
// Column blocks of BN (64 to 128) cover the F*N columns; the u tile is read once per tile
// for all of them.
//
// What bounds it: the FMA pipes (70 % busy at N = 120; the 8 x 8 outer product alone, from
// shared memory, reaches 63 TFLOP/s of the 80.5 derived).  The rest must stay out of its way:
//   multiply-adds packed in pairs along the columns (f32x2): the pipes take as long, but half
//                 the issue slots are left for everything else.  Without the next point
//                 they gained nothing.
//   D^T chunks    neighbouring lanes read neighbouring j of one D row (BK lanes per row, 32 /
//                 BK rows per request).  One column per two lanes, as this kernel had it,
//                 touched 16 rows per request and kept the load/store pipe busy for about as
//                 long as the FMAs themselves.
//   chunk length  16 j (one barrier per 16) beats 8: N = 120, node-major, 617 against 668 us.
//   stores        neighbouring threads hold neighbouring values of the output's contiguous
//                 axis.  Where 16-byte stores are aligned each thread's quads are four
//                 consecutive values; otherwise the positions are permuted so that a quad is
//                 every T-th value (T threads along that axis) and each 4-byte store of a
//                 warp writes runs of T consecutive values.
// Measured before -> after: N = 120, F = 3, E = 310977 node-major 889 -> 603 us; N = 165, F = 3,
// E = 564445 element-major 2584 -> 2114 us; N = 84, F = 4, E = 2^20 element-major 1790 -> 1565 us,
// node-major 1342 us (45 to 50 TFLOP/s with the padding counted).
#include <cuda_runtime.h>

#include "lc_internal.h"
#include "tma.cuh"

namespace lc {

// 4-byte asynchronous copy global -> shared; `bytes` 0 writes a zero (nothing is read).
__device__ __forceinline__ void cp_async4(float *dst, const float *src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(bytes)
                 : "memory");
}

// 16-byte asynchronous copy; the first `bytes` (0..16) come from src, the rest are zeros.
__device__ __forceinline__ void cp_async16(float *dst, const float *src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int BM, int BK, int BN>
struct KsShape {
    static constexpr int TX = BN / 8;        // threads along the columns
    static constexpr int TY = BM / 8;        // threads along the elements
    static constexpr int TH = TX * TY;       // threads of the CTA
    static constexpr int LDA = BM + 4;       // u tile row (one j): BM positions, padded
    static constexpr int LDB = BN + 4;       // D^T chunk row (one j): BN positions, padded
    static constexpr int PP = TH / BK;       // column positions one pass of the CTA's threads copies
    static constexpr int QB = BN / PP;       // passes over a chunk
    static_assert(TH % BK == 0 && BN % PP == 0, "a chunk is copied in whole passes");
};

// The value (0 .. 8T - 1) a position of a tile row holds, for T threads along the row that read
// the quads 4t .. 4t + 3 of each half.  Permuted: thread t's quad is t, t + T, t + 2T, t + 3T.
template <int T>
__device__ __forceinline__ int ks_value(int p, bool perm)
{
    if (!perm)
        return p;
    const int h = p / (4 * T), q = p - h * 4 * T;
    return h * 4 * T + q / 4 + (q % 4) * T;
}
// The inverse: the position of value v.
template <int T>
__device__ __forceinline__ int ks_position(int v, bool perm)
{
    if (!perm)
        return v;
    const int h = v / (4 * T), q = v - h * 4 * T;
    return h * 4 * T + (q % T) * 4 + q / T;
}

// Copy the u tile of elements e0 .. e0+BM-1 into ut[j][position of e] (j < Kp; zeros past N or E).
template <int LAYOUT, int BM, int BK, int BN>
__device__ __forceinline__ void ks_load_u(const KsArgs &a, float *ut, long long e0, int tid)
{
    using S = KsShape<BM, BK, BN>;
    const int N = a.N, Kp = a.Kp;
    const long long E = a.E;
    if (LAYOUT == LC_LAYOUT_NODE_MAJOR) {
        // rows j of u[N][E] are contiguous in e: 16-byte pieces when E % 4 == 0
        if (a.vec_u) {
            constexpr int Q = BM / 4;
            for (int idx = tid; idx < Kp * Q; idx += S::TH) {
                const int j = idx / Q, e = (idx - j * Q) * 4;
                const long long left = E - (e0 + e);
                const uint32_t bytes = (j < N && left > 0) ? (uint32_t)(left >= 4 ? 16 : left * 4) : 0u;
                cp_async16(ut + j * S::LDA + e, bytes ? a.u + (size_t)j * E + e0 + e : a.u, bytes);
            }
        } else {
            for (int idx = tid; idx < Kp * BM; idx += S::TH) {
                const int j = idx / BM, e = idx - j * BM;
                const bool ok = j < N && e0 + e < E;
                cp_async4(ut + j * S::LDA + ks_position<S::TY>(e, !a.vec_out), ok ? a.u + (size_t)j * E + e0 + e : a.u,
                          ok ? 4u : 0u);
            }
        }
    } else {
        // rows e of u[E][N] are contiguous in j: j fastest across threads (coalesced reads),
        // written transposed; the walk idx = e * Kp + j advances by TH without divisions
        const int de = S::TH / Kp, dj = S::TH - de * Kp;
        int e = tid / Kp, j = tid - e * Kp;
        while (e < BM) {
            const bool ok = j < N && e0 + e < E;
            cp_async4(ut + j * S::LDA + e, ok ? a.u + (e0 + e) * N + j : a.u, ok ? 4u : 0u);
            e += de;
            j += dj;
            if (j >= Kp) {
                j -= Kp;
                ++e;
            }
        }
    }
}

// The D^T chunks of one column block.  D read as [F*N][N] has one row per column of D^T.  Lane ->
// (k = tid % BK, position tid / BK + PP q): BK consecutive j of a row per 32 / BK positions.  What
// depends on the column block only is kept from chunk to chunk: per copy an add and a select
// remain (computing the columns in every chunk cost 20 integer instructions a copy).
template <int BM, int BK, int BN>
struct KsB {
    using S = KsShape<BM, BK, BN>;
    int off[S::QB];  // the copy's D offset in the block's first chunk (0 past the last column)
    uint32_t valid;  // bit q: the copy's column exists

    __device__ __forceinline__ void block(const KsArgs &a, int cb, int tid, bool perm)
    {
        const int k = min(tid % BK, a.N - 1), p0 = tid / BK;
        valid = 0;
#pragma unroll
        for (int q = 0; q < S::QB; ++q) {
            const int c = cb * BN + ks_value<S::TX>(p0 + S::PP * q, perm);
            off[q] = c < a.C ? c * a.N + k : 0;
            valid |= (c < a.C ? 1u : 0u) << q;
        }
    }
    // rows kc*BK .. kc*BK+BK-1 into bs[k][position], zeros past N or past the last column
    __device__ __forceinline__ void load(const KsArgs &a, float *bs, int kc, int tid) const
    {
        const int k = tid % BK;
        const bool in = kc * BK + k < a.N;
        const uint32_t ok = in ? valid : 0u;
        const float *src = a.D + (in ? kc * BK : 0);
        float *dst = bs + k * S::LDB + tid / BK;
#pragma unroll
        for (int q = 0; q < S::QB; ++q)
            cp_async4(dst + S::PP * q, src + off[q], (ok >> q & 1u) * 4u);
    }
};

template <int LAYOUT, int BM, int BK, int BN>
__global__ void __launch_bounds__(KsShape<BM, BK, BN>::TH, BM == 128 ? 2 : 3)
    ks_contract_kernel(const __grid_constant__ KsArgs a)
{
    using S = KsShape<BM, BK, BN>;
    constexpr bool NODE = LAYOUT == LC_LAYOUT_NODE_MAJOR;
    extern __shared__ __align__(16) float ks_smem[];
    const int N = a.N, Kp = a.Kp, nkc = a.nkc, nb = a.nblocks;
    const long long E = a.E;
    float *ubuf = ks_smem;                                    // [ubufs][Kp][LDA]
    float *bbuf = ks_smem + (size_t)a.ubufs * Kp * S::LDA;    // [2][BK][LDB]
    // the threads of a warp run along the output's contiguous axis
    const int tid = threadIdx.x;
    const int tx = NODE ? tid / S::TY : tid % S::TX, ty = NODE ? tid % S::TY : tid / S::TX;
    const bool permc = !NODE && !a.vec_out;  // column positions permuted (element-major, N % 4 != 0)
    const long long t0 = blockIdx.x, dt = gridDim.x;
    if (t0 >= a.ntiles)
        return;

    uint64_t acc2[8][4];  // acc2[x][p]: columns 2p and 2p + 1 of the thread's eight, packed
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int p = 0; p < 4; ++p)
            acc2[x][p] = 0;

    // prologue: the first tile's u and the first chunk
    ks_load_u<LAYOUT, BM, BK, BN>(a, ubuf, t0 * BM, tid);
    KsB<BM, BK, BN> bsrc;
    bsrc.block(a, 0, tid, permc);
    bsrc.load(a, bbuf, 0, tid);
    cp_async_commit();
    int sl = 0;  // ring slot of the current chunk
    int ti = 0;
    for (long long t = t0; t < a.ntiles; t += dt, ++ti) {
        const long long e0 = t * BM;
        const int ub = a.ubufs == 2 ? (ti & 1) : 0;
        const float *ut = ubuf + (size_t)ub * Kp * S::LDA;
        const bool has_next_tile = t + dt < a.ntiles;
        for (int cb = 0; cb < nb; ++cb) {
            for (int kc = 0; kc < nkc; ++kc) {
                cp_async_wait_all();  // this thread's copies of the current chunk (and tile) landed
                __syncthreads();      // everyone's landed; everyone is done with the other slot
                if (a.ubufs == 1 && ti > 0 && cb == 0 && kc == 0) {
                    // one u buffer: the previous tile's reads are over only now
                    ks_load_u<LAYOUT, BM, BK, BN>(a, ubuf, e0, tid);
                    cp_async_commit();
                    cp_async_wait_all();
                    __syncthreads();
                }
                // the next chunk: (cb, kc + 1), (cb + 1, 0) or the next tile's (0, 0)
                int nkc_ = kc + 1, ncb = cb;
                if (nkc_ == nkc) {
                    nkc_ = 0;
                    ncb = cb + 1;
                }
                if (ncb < nb || has_next_tile) {
                    if (nkc_ == 0 && nb > 1)
                        bsrc.block(a, ncb == nb ? 0 : ncb, tid, permc);
                    bsrc.load(a, bbuf + (size_t)(sl ^ 1) * BK * S::LDB, nkc_, tid);
                }
                if (a.ubufs == 2 && cb == 0 && kc == 0 && has_next_tile)
                    ks_load_u<LAYOUT, BM, BK, BN>(a, ubuf + (size_t)(ub ^ 1) * Kp * S::LDA, (t + dt) * BM, tid);
                cp_async_commit();

                const float *A = ut + (size_t)kc * BK * S::LDA + 4 * ty;
                const float *B = bbuf + (size_t)sl * BK * S::LDB + 4 * tx;
#pragma unroll
                for (int k = 0; k < BK; ++k) {
                    if (BK == 16 && k == 8 && kc * BK + 8 >= N)
                        break;  // the last chunk's second half holds no node
                    const float4 a0 = *reinterpret_cast<const float4 *>(A + k * S::LDA);
                    const float4 a1 = *reinterpret_cast<const float4 *>(A + k * S::LDA + BM / 2);
                    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(B + k * S::LDB);
                    const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(B + k * S::LDB + BN / 2);
                    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                    const uint64_t bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const uint64_t ax = pack_f32x2(av[x], av[x]);
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            acc2[x][p] = fma_f32x2(ax, bv[p], acc2[x][p]);
                    }
                }
                sl ^= 1;
            }
            float acc[8][8];
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float2 v = unpack_f32x2(acc2[x][p]);
                    acc[x][2 * p] = v.x;
                    acc[x][2 * p + 1] = v.y;
                    acc2[x][p] = 0;
                }
            // store the 8 x 8 block: acc[4g + z][4h + y] is element e0 + g BM/2 + .., column
            // cb BN + h BN/2 + ..
            if (NODE) {
                // out[f][i][e] = column c, contiguous in e
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        const int c = cb * BN + h * (BN / 2) + 4 * tx + y;
                        if (c >= a.C)
                            break;
                        float *col = a.out + (size_t)c * E;  // (f N + i) E
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            const float vv[4] = {acc[4 * g][4 * h + y], acc[4 * g + 1][4 * h + y],
                                                 acc[4 * g + 2][4 * h + y], acc[4 * g + 3][4 * h + y]};
                            const long long eb = e0 + g * (BM / 2);
                            if (a.vec_out) {
                                // E % 4 == 0: a quad is inside or outside
                                if (eb + 4 * ty < E)
                                    *reinterpret_cast<float4 *>(col + eb + 4 * ty) =
                                        make_float4(vv[0], vv[1], vv[2], vv[3]);
                            } else {
#pragma unroll
                                for (int z = 0; z < 4; ++z)
                                    if (eb + ty + z * S::TY < E)
                                        col[eb + ty + z * S::TY] = vv[z];
                            }
                        }
                    }
            } else if (a.vec_out) {
                // out[f][e][i], N % 4 == 0: four consecutive columns of one operator
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c4 = cb * BN + h * (BN / 2) + 4 * tx;
                    if (c4 >= a.C)
                        continue;
                    const int f4 = c4 / N, i4 = c4 - f4 * N;
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const long long e = e0 + (x / 4) * (BM / 2) + 4 * ty + x % 4;
                        if (e < E)
                            *reinterpret_cast<float4 *>(a.out + ((size_t)f4 * E + e) * N + i4) =
                                make_float4(acc[x][4 * h], acc[x][4 * h + 1], acc[x][4 * h + 2], acc[x][4 * h + 3]);
                    }
                }
            } else {
                // out[f][e][i], permuted columns: c, c + TX, c + 2 TX, c + 3 TX
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        const int c = cb * BN + h * (BN / 2) + tx + y * S::TX;
                        if (c >= a.C)
                            break;
                        const int f = c / N, i = c - f * N;
                        float *o = a.out + ((size_t)f * E + e0 + 4 * ty) * N + i;
#pragma unroll
                        for (int x = 0; x < 8; ++x) {
                            const int de = (x / 4) * (BM / 2) + x % 4;
                            if (e0 + 4 * ty + de < E)
                                o[de * N] = acc[x][4 * h + y];
                        }
                    }
            }
        }
    }
    cp_async_wait_all();  // no copy outlives the CTA
}

// Column block width: the one of the compiled widths that covers C columns soonest.
int ks_block_cols(int C, int bm)
{
    if (bm != 128)
        return 128;
    // Time per padded column, in hundredths of a block of 128's (measured, N = 64 to 95: 160 us a unit
    // of work, 174, 188, 211, ...): a smaller block has fewer warps to hide latency with, and 80 and 112
    // do not deal them evenly to the four schedulers.  N = 75, F = 3, E = 177780: 255 us with 3 x 80
    // columns, 198 with 2 x 128; N = 73, F = 4, E = 140742: 261 with 4 x 80, 229 with 3 x 112.
    const int width[] = {128, 112, 96, 80, 64}, weight[] = {100, 108, 118, 132, 145};
    int best = 0;
    auto cost = [&](int q) { return (C + width[q] - 1) / width[q] * width[q] * weight[q]; };
    for (int q = 1; q < 5; ++q)
        if (cost(q) < cost(best))
            best = q;
    return width[best];
}

// Length of the j chunks: 16, but 8 where two CTAs of 128 elements then fit an SM and with 16 only one
// (N = 177 to 200; N = 200, F = 1, E = 100001: 309 -> 282 us).
int ks_chunk(int N, int F, int bm)
{
    if (bm != 128)
        return 16;
    const size_t two = 232448 / 2 - 1024;  // (1 KB reserved per CTA)
    auto bytes = [&](int bk) { return ks_smem_bytes((N + bk - 1) / bk * bk, bm, bk, ks_block_cols(F * N, bm), 1); };
    return bytes(16) > two && bytes(8) <= two ? 8 : 16;
}

int ks_threads(int bm, int bn) { return (bm / 8) * (bn / 8); }

size_t ks_smem_bytes(int Kp, int bm, int bk, int bn, int ubufs)
{
    return sizeof(float) * ((size_t)ubufs * Kp * (bm + 4) + 2 * (size_t)bk * (bn + 4));
}

template <int LAYOUT, int BK>
static void *ks_fn128(int bn)
{
    switch (bn) {
    case 64: return reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 128, BK, 64>);
    case 80: return reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 128, BK, 80>);
    case 96: return reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 128, BK, 96>);
    case 112: return reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 128, BK, 112>);
    default: return reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 128, BK, 128>);
    }
}

template <int LAYOUT>
static void *ks_fn(int bm, int bk, int bn)
{
    if (bm == 128)
        return bk == 16 ? ks_fn128<LAYOUT, 16>(bn) : ks_fn128<LAYOUT, 8>(bn);
    return bk == 16 ? reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 64, 16, 128>)
                    : reinterpret_cast<void *>(&ks_contract_kernel<LAYOUT, 64, 8, 128>);
}

lc_status ks_launch(const KsArgs &a, int layout, int bm, int bk, int grid, cudaStream_t s, bool set_attr)
{
    if (!(bm == 64 || bm == 128) || !(bk == 8 || bk == 16))
        return LC_ERR_INVALID_VARIANT;
    void *fn = layout == LC_LAYOUT_NODE_MAJOR ? ks_fn<LC_LAYOUT_NODE_MAJOR>(bm, bk, a.bn)
                                              : ks_fn<LC_LAYOUT_ELEM_MAJOR>(bm, bk, a.bn);
    const size_t smem = ks_smem_bytes(a.Kp, bm, bk, a.bn, a.ubufs);
    cudaError_t e = cudaSuccess;
    if (set_attr) {
        e = allow_smem(fn);
        if (e != cudaSuccess)
            return cuda_fail(e);
    }
    if (grid <= 0)
        return LC_OK;  // attribute set only (a capture launches later)
    KsArgs args = a;
    void *params[] = {&args};
    e = cudaLaunchKernel(fn, dim3(grid), dim3(ks_threads(bm, a.bn)), params, smem, s);
    return e == cudaSuccess ? LC_OK : cuda_fail(e);
}

}  // namespace lc
