// Row kernel (FP32, 13 <= N <= 40): the SIMT engine's form with the j loop wholly unrolled
// (descriptor unroll 8 with prefetch_smem 1), for
//     out[f,e,i] = sum_j D[f,i,j] * u[e,j]                (dG FEM volume, Table 1)
//
// A thread keeps the whole rows u[e][:] of EPT = 4 (or 2) elements in registers, packed in pairs
// along j, and runs over the output columns four at a time; the operator rows come from shared
// memory, the same 16 bytes for every lane of the warp.  Such a read still writes 512 bytes of
// registers, four cycles of the SM's load path, and feeds 2 EPT packed multiply-adds (f32x2, half
// a cycle of the SM each): with EPT = 4 the two take equally long, with EPT = 2 the reads bound
// the kernel (N = 35, F = 3, E = 2^21: 368 us).  The 4 x 8 register blocks of the tiled kernel
// (simt.cuh) ran at 0.38 of the FMA rate there (494 us).  The two halves of a packed sum (even j,
// odd j) are added at the end: a pairwise sum, whose rounding error is below the plain chain's
// (8.2e-8 against 1.1e-7).
//
// Warps are on their own (no CTA barrier after the operators are staged): a warp takes chunks of
// 32 EPT elements (lane l: elements l, l + 32, ...).
//   element-major  each warp has one or two buffers of the chunk's rows; the bulk-copy engine
//                  fetches u rows into one, each operator's outputs are staged in a free one and
//                  written by the bulk-copy engine as one contiguous run.  With two buffers the
//                  next chunk's rows come while the last operator is computed; with one (two do
//                  not fit beside eight warps) the SMSP's other warp covers the waits;
//   node-major     u comes straight from global memory (coalesced, all of a chunk's loads in
//                  flight at once, any alignment) and outputs leave registers coalesced.
// EPT = 4 with eight warps above N = 20 where every warp gets a chunk, else EPT = 2 (smaller chunks
// spread a small batch over more SMs); where warps would be left without a chunk, each operator of
// a chunk is a unit of its own.
// Measured, F = 3, E = 2^21, before (simt.cuh) -> after: N = 35 element-major 494 -> 351 us (HBM floor
// 175, FMA floor 191), node-major 486 -> 356; N = 20 280 -> 121 and 228 -> 142 (HBM floor 100).  At
// N = 35 the FMA pipes are 53 % busy, the load/store wavefronts 33 %, and an instruction issues in
// 39 % of the cycles: the largest stall is the fixed latency of a warp's own instructions (two
// warps an SMSP, all the registers allow), then the wait for its next rows.
#include <cuda_runtime.h>

#include <algorithm>

#include "lc_internal.h"
#include "row.cuh"

namespace lc {

// operators: [F N + 3][NP] floats (the column loop reads up to three rows past the last)
__host__ __device__ inline size_t row_d_bytes(int N, int F) { return sizeof(float) * (size_t)(F * N + 3) * row_np(N); }

template <int NP, int LAYOUT, int EPT>
__global__ void __launch_bounds__(EPT == 4 ? 256 : 512, 1) row_contract_kernel(SimtArgs a)
{
    constexpr bool NODE = LAYOUT == LC_LAYOUT_NODE_MAJOR;
    constexpr int CH = 32 * EPT;  // elements of a chunk
    extern __shared__ __align__(16) unsigned char row_smem[];
    const int N = a.N, F = a.F;
    const long long E = a.E;
    const float *__restrict__ D = static_cast<const float *>(a.D);
    const float *__restrict__ u = static_cast<const float *>(a.u);
    float *__restrict__ out = static_cast<float *>(a.out);
    float *Ds = reinterpret_cast<float *>(row_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    // element-major: this warp's NB buffers of CH rows, then the mbarriers of all warps
    const int NB = a.stages;
    const int bufn = CH * N;  // (a multiple of 64 floats: 16-byte aligned)
    unsigned char *rest = row_smem + row_d_bytes(N, F);
    float *buf = reinterpret_cast<float *>(rest) + (size_t)warp * NB * bufn;
    uint64_t *bar = reinterpret_cast<uint64_t *>(rest + sizeof(float) * (size_t)W * NB * bufn) + warp;
    // units of work: (chunk, part): every operator of a chunk, or (P = F) one operator each
    const int P = a.nchunks, nf = F / P;
    const long long nunits = a.ntiles * P, step = (long long)gridDim.x * W;
    const long long first = (long long)warp * gridDim.x + blockIdx.x;  // one warp on every SM before a second

    // rows of unit w's chunk; the bulk engine fetches whole chunks (the last one's bytes may not be a multiple of 16)
    auto chunk_of = [&](long long w) { return P == 1 ? w : w / P; };
    auto rows_of = [&](long long w) { return (int)min((long long)CH, E - chunk_of(w) * CH); };
    auto bulk_ok = [&](int rows) { return ((rows * N) & 3) == 0; };
    auto fetch = [&](long long w, float *to) {  // lane 0
        const int rows = rows_of(w);
        if (bulk_ok(rows)) {
            mbar_arrive_expect_tx(bar, (uint32_t)(rows * N) * 4u);
            bulk_g2s(to, u + chunk_of(w) * CH * N, (uint32_t)(rows * N) * 4u, bar);
        }
    };
    if (!NODE && lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        if (first < nunits)
            fetch(first, buf);
    }
    for (int idx = tid; idx < (F * N + 3) * NP; idx += blockDim.x) {
        const int c = idx / NP, j = idx - c * NP;
        Ds[idx] = c < F * N && j < N ? D[(size_t)c * N + j] : 0.f;
    }
    __syncthreads();

    uint64_t ur[EPT][NP / 2];
    uint32_t phase = 0;
    int cur = 0;  // the buffer that holds the current chunk's rows
    for (long long w = first; w < nunits; w += step) {
        const long long t = chunk_of(w);
        const int f0 = (int)(w - t * P) * nf;  // this unit's operators f0 .. f0 + nf - 1
        const long long e0 = t * CH;
        const int rows = rows_of(w);
        if (NODE) {
            bool in[EPT];
#pragma unroll
            for (int x = 0; x < EPT; ++x)
                in[x] = lane + 32 * x < rows;
            const float *p = u + e0 + lane;
            float v[EPT][NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
#pragma unroll
                for (int x = 0; x < EPT; ++x)
                    v[x][j] = in[x] && j < N ? __ldg(p + 32 * x) : 0.f;
                p += E;
            }
#pragma unroll
            for (int x = 0; x < EPT; ++x)
#pragma unroll
                for (int q = 0; q < NP / 2; ++q)
                    ur[x][q] = pack_f32x2(v[x][2 * q], v[x][2 * q + 1]);
            const int C = (f0 + nf) * N;
            float *o = out + (size_t)f0 * N * E + e0 + lane;
            for (int c = f0 * N; c < C; c += 4) {
                float r[EPT][4];
                row_columns<NP, EPT>(Ds + (size_t)c * NP, ur, r);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (c + m < C) {
#pragma unroll
                        for (int x = 0; x < EPT; ++x)
                            if (in[x])
                                o[32 * x] = r[x][m];
                    }
                    o += E;
                }
            }
            continue;
        }
        float *ub = buf + cur * bufn;
        if (bulk_ok(rows)) {
            if (!mbar_wait(bar, phase)) {
                if (lane == 0)
                    atomicOr(a.err, 1u);
                break;
            }
            phase ^= 1u;
        } else {
            if (lane == 0)
                bulk_wait_read0();
            __syncwarp();
            for (int k = lane; k < rows * N; k += 32)
                ub[k] = u[e0 * N + k];
            __syncwarp();
        }
        // the rows of this lane (rows past the last element hold whatever the buffer does)
#pragma unroll
        for (int x = 0; x < EPT; ++x) {
            const float *p = ub + (lane + 32 * x) * N;
            if ((N & 3) == 0) {
#pragma unroll
                for (int q = 0; q < NP / 4; ++q) {
                    const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(p)[q];
                    ur[x][2 * q] = v.x;
                    ur[x][2 * q + 1] = v.y;
                }
            } else {
                float v[NP];
#pragma unroll
                for (int j = 0; j < NP; ++j)
                    v[j] = j < N ? p[j] : 0.f;
#pragma unroll
                for (int q = 0; q < NP / 2; ++q)
                    ur[x][q] = pack_f32x2(v[2 * q], v[2 * q + 1]);
            }
        }
        __syncwarp();
        const int total = rows * N;
        for (int k = 0; k < nf; ++k) {
            const int f = f0 + k;
            const int ob = NB == 2 ? cur ^ 1 ^ (k & 1) : 0;
            // the store that last read this buffer is done reading it
            if (lane == 0) {
                if (k == 0 || NB == 1)
                    bulk_wait_read0();
                else if (k >= 2)
                    bulk_wait_read(1);
            }
            __syncwarp();
            float *o0 = buf + ob * bufn + lane * N;
            const float *dp = Ds + (size_t)f * N * NP;
            const int half = (N / 2) & ~3;
            for (int i = 0; i < N; i += 4) {
                float r[EPT][4];
                row_columns<NP, EPT>(dp + (size_t)i * NP, ur, r);
#pragma unroll
                for (int x = 0; x < EPT; ++x) {
                    float *o = o0 + 32 * x * N + i;
                    if ((N & 3) == 0) {
                        *reinterpret_cast<float4 *>(o) = make_float4(r[x][0], r[x][1], r[x][2], r[x][3]);
                    } else {
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (i + m < N)
                                o[m] = r[x][m];
                    }
                }
                // in the middle of the last operator: every row of u has been used (the columns before
                // this one needed them), and the other buffer's store has had time to be read
                if (NB == 2 && k == nf - 1 && i == half && lane == 0) {
                    bulk_wait_read0();
                    if (w + step < nunits)
                        fetch(w + step, buf + (ob ^ 1) * bufn);
                }
            }
            float *dst = out + ((size_t)f * E + e0) * N;
            const float *src = buf + ob * bufn;
            if (a.bulk_store && (total & 3) == 0) {
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    bulk_s2g(dst, src, (uint32_t)total * 4u);
                    bulk_commit();
                }
            } else {
                __syncwarp();
                for (int q = lane; q < total; q += 32)
                    dst[q] = src[q];
                fence_async_smem();  // a later bulk copy may write this buffer
                __syncwarp();
            }
        }
        if (NB == 2) {
            cur = cur ^ 1 ^ ((nf - 1) & 1) ^ 1;  // the buffer the last operator left free
        } else if (lane == 0 && w + step < nunits) {
            bulk_wait_read0();
            fetch(w + step, buf);
        }
    }
    if (!NODE && lane == 0)
        bulk_wait0();
}

// Elements a thread, warps a CTA and buffers a warp (0 warps: it does not fit).
RowPlan row_plan(long long E, int N, int F, bool node, int sms, size_t smem_cap)
{
    RowPlan p{};
    const size_t d = row_d_bytes(N, F);
    if (d > smem_cap)
        return p;
    auto per = [&](int ept, int nb) { return nb * sizeof(float) * (size_t)(32 * ept) * N + sizeof(uint64_t); };
    p.ept = N > 20 && E >= 128ll * 8 * sms ? 4 : 2;  // (up to N = 20 HBM bounds it: two elements, twice the warps)
    const int most = p.ept == 4 ? 8 : 16;
    p.buffers = node || d + most * per(p.ept, 2) <= smem_cap || p.ept == 2 ? 2 : 1;
    p.warps = node ? most : (int)std::min<size_t>(most, (smem_cap - d) / per(p.ept, p.buffers));
    // a batch that would leave warps without a chunk: one operator a unit (the chunk is read F times)
    p.parts = (E + 32 * p.ept - 1) / (32 * p.ept) < (long long)p.warps * sms ? F : 1;
    p.smem = d + (node ? 0 : p.warps * per(p.ept, p.buffers));
    return p;
}

template <int LAYOUT, int EPT>
static void *row_fn(int np)
{
    switch (np) {
    case 16: return reinterpret_cast<void *>(&row_contract_kernel<16, LAYOUT, EPT>);
    case 20: return reinterpret_cast<void *>(&row_contract_kernel<20, LAYOUT, EPT>);
    case 24: return reinterpret_cast<void *>(&row_contract_kernel<24, LAYOUT, EPT>);
    case 28: return reinterpret_cast<void *>(&row_contract_kernel<28, LAYOUT, EPT>);
    case 32: return reinterpret_cast<void *>(&row_contract_kernel<32, LAYOUT, EPT>);
    case 36: return reinterpret_cast<void *>(&row_contract_kernel<36, LAYOUT, EPT>);
    case 40: return reinterpret_cast<void *>(&row_contract_kernel<40, LAYOUT, EPT>);
    default: return nullptr;
    }
}

lc_status row_launch(const SimtArgs &a, int layout, int ept, int grid, int threads, size_t smem, cudaStream_t s)
{
    const int np = row_np(a.N);
    void *fn = layout == LC_LAYOUT_NODE_MAJOR
                   ? (ept == 4 ? row_fn<LC_LAYOUT_NODE_MAJOR, 4>(np) : row_fn<LC_LAYOUT_NODE_MAJOR, 2>(np))
                   : (ept == 4 ? row_fn<LC_LAYOUT_ELEM_MAJOR, 4>(np) : row_fn<LC_LAYOUT_ELEM_MAJOR, 2>(np));
    if (!fn)
        return LC_ERR_INVALID_VARIANT;
    cudaError_t e = allow_smem(fn);
    if (e != cudaSuccess)
        return cuda_fail(e);
    SimtArgs args = a;
    void *params[] = {&args};
    e = cudaLaunchKernel(fn, dim3(grid), dim3(threads), params, smem, s);
    return e == cudaSuccess ? LC_OK : cuda_fail(e);
}

}  // namespace lc
