// Surface lift with the flux rows in registers (Nf <= 4, M = Nf * Nfp <= kLiftRowMaxM):
//     out[e,i] (+)= sum_m L[i,m] * flux[e,m],  flux[e,m] = s[e,m/Nfp] * (u[e,fmask[m]] - u_flat[vmapP[e,m]])
//
// Lanes l and l + 16 of a warp share EPT elements: the first gathers the fluxes of the lower half of
// the face nodes straight into registers, packed in pairs along m, the second those of the upper half.
// Each runs over the output columns four at a time against its half of the rows of L in shared memory
// (row.cuh); one shuffle per two outputs adds the halves.  No flux tile, no transposition and no
// barrier between the gather and the products; warps only share the u window.
//   window   the rows of the CTA's tile and `halo` rows on either side, fetched by the bulk-copy
//            engine; nothing reads it after the gather, so the next tile's window comes during the
//            products, issued by the warp that is last to finish its gather;
//   indexes  a warp's vmapP rows (and face scales where they fit), fetched by the bulk-copy engine
//            into its own two buffers: A (the first 32 rows; refilled during the products) and B (the
//            others), which is also where the outputs are staged for one contiguous bulk store, and
//            which is refilled when that store has been read, while A is being gathered.
// An exterior trace outside the window is fetched from global memory ahead of the row's gather and
// parked over its index; an index out of range gives NaN there and sets the error word.
//
// What bounds it: shared memory and the FMA pipes together.  A read of L, the same 16 bytes for the
// lanes of a half, costs four cycles of the SM's load path and feeds eight packed multiply-adds (four
// cycles); with whole rows a lane and two elements it fed four, and the reads were the bound (355 us
// below).  At degree 4 (N = 35, M = 60) a tile of 512 elements takes about 24600 cycles: products
// 13000 (FMA floor 9200), gather 8800, staging and stores 1200.  The gather's loads stand in a row
// with nothing conditional between them: with the change of face tested in that loop it took 13000.
// Measured against the tiled kernel (lift.cu), us: degree 4, E = 2^21 605 -> 325 (HBM floor 168),
// accumulating 1105 -> 470 (with 45 for clearing out); degree 3 408 -> 173 (105); degree 2 302 -> 118
// (60; rows of N = 10 and 20 values meet in the same banks); degree 1, E = 1000003 122 -> 45; degree
// 4, E = 100003 with neighbours 200 elements away 44 -> 31, E = 4099 12.8 -> 11.4.
#include <cuda_runtime.h>

#include <algorithm>

#include "lc_internal.h"
#include "row.cuh"

namespace lc {

static constexpr int kLiftRowWarps = 8;
static constexpr int kLiftRowMaxM = 64;
// Face nodes of a half, padded to whole 16-byte reads.
__host__ __device__ constexpr int lift_row_half(int M) { return (M + 7) / 8 * 4; }
// Elements a lane pair shares: six where their fluxes leave registers to spare, else four; two (for
// more and smaller chunks) in a batch that gives no SM more than three such chunks.
// (degree 3, E = 12000: 13.4 us with six, 11.6 with two)
__host__ __device__ constexpr int lift_row_ept(int MH) { return MH <= 20 ? 6 : 4; }

// Shared memory: L rows [N to a multiple of 4][2 MH], node of each face node [2 MH], the u window, per
// warp the buffers A and B, the barriers (the window's, a counter, two per warp).
struct LiftRowSmem {
    size_t fnode, win, warp, a_bytes, per_warp, bars, total;
};
__host__ __device__ inline LiftRowSmem lift_row_smem(int N, int M, int Nf, int ept, int warps, int halo, int stage_s)
{
    LiftRowSmem s;
    const int MH = lift_row_half(M), CH = 16 * ept;
    s.fnode = sizeof(float) * (size_t)row_np(N) * 2 * MH;
    s.win = s.fnode + sizeof(int) * 2 * (size_t)MH;
    s.warp = s.win + sizeof(float) * (size_t)(CH * warps + 2 * halo) * N;  // (a multiple of 4 rows)
    const size_t row = sizeof(int) * (size_t)(M + (stage_s ? Nf : 0));
    s.a_bytes = 32 * row;
    const size_t b_rows = (CH - 32) * row, b_out = sizeof(float) * (size_t)CH * N;
    s.per_warp = s.a_bytes + (b_rows > b_out ? b_rows : b_out);
    s.bars = s.warp + s.per_warp * warps;
    s.total = s.bars + sizeof(uint64_t) * (2 + 2 * (size_t)warps);
    return s;
}

// A shared-memory load by 32-bit address, in program order with the waits around it.
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int MH, int EPT, bool LINES>  // LINES: M = 2 MH is a multiple of 32
__global__ void __launch_bounds__(32 * kLiftRowWarps, 1) lift_row_kernel(LiftArgs a)
{
    constexpr int CH = 16 * EPT;  // elements of a warp's chunk
    extern __shared__ __align__(16) unsigned char lift_row_buf[];
    const int N = a.N, M = a.M, Nfp = a.Nfp, Nf = a.Nf, H = a.halo;
    const int E = (int)a.E;  // E * N < 2^31
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = a.warps;
    const int half = lane >> 4, m0 = half * MH;  // this lane's face nodes m0 .. m0 + MH - 1
    const LiftRowSmem lay = lift_row_smem(N, M, Nf, EPT, W, H, a.stage_s);
    float *Ls = reinterpret_cast<float *>(lift_row_buf);
    int *fnode = reinterpret_cast<int *>(lift_row_buf + lay.fnode);
    float *win = reinterpret_cast<float *>(lift_row_buf + lay.win);
    unsigned char *mine = lift_row_buf + lay.warp + (size_t)warp * lay.per_warp;
    int *vA = reinterpret_cast<int *>(mine), *vB = reinterpret_cast<int *>(mine + lay.a_bytes);
    float *stage = reinterpret_cast<float *>(vB);
    uint64_t *wbar = reinterpret_cast<uint64_t *>(lift_row_buf + lay.bars);
    unsigned int *gathered = reinterpret_cast<unsigned int *>(wbar + 1);
    uint64_t *abar = wbar + 2 + 2 * warp, *bbar = abar + 1;
    const int TE = CH * W;
    const int ntiles = (E + TE - 1) / TE;

    // rows of this warp's chunk of tile t (none: <= 0)
    auto rows_of = [&](int t) { return warp < W ? min(CH, E - t * TE - warp * CH) : 0; };
    // lane 0: rows r0 .. r0 + cap - 1 of the chunk into v (a part below 16 bytes at the end is left out)
    auto fetch = [&](int t, int *v, uint64_t *bar, int r0, int cap) {
        const int n = min(rows_of(t) - r0, cap);
        if (n <= 0)
            return;
        const long long e = (long long)t * TE + warp * CH + r0;
        const uint32_t vb = (uint32_t)(n * M * 4) & ~15u, sb = a.stage_s ? (uint32_t)(n * Nf * 4) & ~15u : 0u;
        mbar_arrive_expect_tx(bar, vb + sb);
        if (vb)
            bulk_g2s(v, a.vmapP + e * M, vb, bar);
        if (sb)
            bulk_g2s(v + cap * M, a.s + e * Nf, sb, bar);
    };
    // the warp: wait for them and add the left-out part
    auto arrived = [&](int t, int *v, uint64_t *bar, uint32_t phase, int r0, int cap) {
        const int n = min(rows_of(t) - r0, cap);
        if (n <= 0)
            return true;
        const bool ok = mbar_wait(bar, phase);
        if (((n * M | n * Nf) & 3) != 0) {
            const long long e = (long long)t * TE + warp * CH + r0;
            const int q = (n * M & ~3) + lane, p = (n * Nf & ~3) + lane;
            if (q < n * M)
                v[q] = a.vmapP[e * M + q];
            if (a.stage_s && p < n * Nf)
                v[cap * M + p] = __float_as_int(a.s[e * Nf + p]);
            __syncwarp();
        }
        return ok;
    };
    // scales that are not staged: on their way to L1
    auto scales = [&](int t) {
        if (!a.stage_s)
            for (int r = lane; r < rows_of(t); r += 32)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(a.s + ((long long)t * TE + warp * CH + r) * Nf));
    };
    auto window = [&](int t) {  // one thread
        const int lo = max(0, t * TE - H), hi = min(E, t * TE + TE + H);
        const uint32_t bytes = (uint32_t)((hi - lo) * N * 4) & ~15u;
        mbar_arrive_expect_tx(wbar, bytes);
        if (bytes)
            bulk_g2s(win, a.u + (long long)lo * N, bytes, wbar);
    };
    if (tid == 0) {
        mbar_init(wbar, 1);
        for (int w = 0; w < 2 * W; ++w)
            mbar_init(wbar + 2 + w, 1);
        *gathered = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0)
        window(blockIdx.x);
    if (lane == 0) {
        fetch(blockIdx.x, vA, abar, 0, 32);
        fetch(blockIdx.x, vB, bbar, 32, CH - 32);
    }
    scales(blockIdx.x);
    const int NL = row_np(N);
#pragma unroll 8
    for (int idx = tid; idx < NL * 2 * MH; idx += blockDim.x) {
        const int i = idx / (2 * MH), m = idx - i * 2 * MH;
        Ls[idx] = i < N && m < M ? __ldg(a.L + (size_t)i * M + m) : 0.f;
    }
    for (int m = tid; m < 2 * MH; m += blockDim.x) {
        const int j = m < M ? a.fmask[m] : 0;
        const bool bad = j < 0 || j >= N;
        fnode[m] = bad ? 0 : 4 * j;  // (bytes) out of range: recorded, node 0 read instead
        if (bad)
            atomicOr(a.err, 2u);
    }
    __syncthreads();
    const int b1 = Nfp - m0, b2 = 2 * Nfp - m0, b3 = 3 * Nfp - m0;  // where this lane's nodes change face
    const uint32_t win_s = smem_addr(win);

    uint64_t fx[EPT][MH / 2];
    uint32_t phase = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, phase ^= 1u) {
        const int e0 = t * TE, lo = max(0, e0 - H), hi = min(E, e0 + TE + H);
        const int rows = rows_of(t), nt = t + (int)gridDim.x;
        const int wn = (hi - lo) * N, wb = lo * N;
        if (!mbar_wait(wbar, phase)) {
            if (lane == 0)
                atomicOr(a.err, 1u);
            break;
        }
        if (rows <= 0)
            break;  // (the last tile, or a warp that only helped to lay out L)
        if ((wn & 3) != 0) {  // the part below 16 bytes at the end (each warp writes the same values)
            const int q = (wn & ~3) + lane;
            if (q < wn)
                win[q] = a.u[wb + q];
            fence_async_smem();  // (a bulk copy may write the window again)
            __syncwarp();
        }
        unsigned int seen = 0;
        bool ok = true, parked = false;
#pragma unroll
        for (int x = 0; x < EPT; ++x) {
            if (x == 0)
                ok = arrived(t, vA, abar, phase, 0, 32);
            else if (x == 2)
                ok = arrived(t, vB, bbar, phase, 32, CH - 32) && ok;
            // slots 2k and 2k + 1: this lane's element of each 32, then its partner's (one shuffle of
            // the odd slot's sums then gives each lane its own element's other half)
            const int r = (x / 2) * 32 + ((x & 1) ? lane ^ 16 : lane);
            const bool live = r < rows;
            const int rr = live ? r : 0;  // (no such element: row 0, whose result is not used)
            int *v0 = rr < 32 ? vA : vB;
            int *vr = v0 + (rr < 32 ? rr : rr - 32) * M + m0;
            const float *sp = a.stage_s ? reinterpret_cast<const float *>(v0 + (rr < 32 ? 32 : CH - 32) * M) +
                                              (rr < 32 ? rr : rr - 32) * Nf
                                        : a.s + ((long long)e0 + warp * CH + rr) * Nf;
            float sv[4];
            if (Nf == 4) {
                const float4 v = *reinterpret_cast<const float4 *>(sp);
                sv[0] = v.x, sv[1] = v.y, sv[2] = v.z, sv[3] = v.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    sv[k] = sp[min(k, Nf - 1)];
            }
            int q[MH];
            unsigned int far = 0;
            if ((M & 3) == 0) {
#pragma unroll
                for (int m = 0; m < MH; m += 4) {
                    const int4 v = *reinterpret_cast<const int4 *>(vr + m);
                    q[m] = v.x - wb, q[m + 1] = v.y - wb, q[m + 2] = v.z - wb, q[m + 3] = v.w - wb;
                }
            } else {
#pragma unroll
                for (int m = 0; m < MH; ++m)
                    q[m] = vr[m] - wb;
            }
#pragma unroll
            for (int m = 0; m < MH; ++m) {
                if (m >= MH - 8 && m0 + m >= M)
                    q[m] = 0;  // (padding: 2 MH - 8 < M)
                far = max(far, (unsigned int)q[m]);
            }
            if constexpr (LINES) {
                // Index rows of whole 128-byte lines: lanes that each walk their own row would meet in one
                // bank, and so they take the far halves together, a row's half over neighbouring lanes (two
                // where 16 lanes cover it).  (N = 24, M = 64, E = 1000003, 1000 away: 619 -> 352 us; for
                // other M a row a lane is as fast or faster, degree 4 273 against 353.)
                unsigned int left = __ballot_sync(0xffffffffu, far >= (unsigned int)wn);
                if (left != 0) {
                    parked = true;
                    left &= __ballot_sync(0xffffffffu, live);
                    constexpr int P = MH <= 16 ? 2 : 1;
                    const int sub = lane / (32 / P), m = lane % (32 / P);
                    int *base = x < 2 ? vA : vB + (x / 2 - 1) * 32 * M;
                    for (int o0 = 0; o0 < 32; o0 += 8 * P) {
                        if ((left >> o0 & (0xffffffffu >> (32 - 8 * P))) == 0)
                            continue;
                        float v[8];
                        int at[8];
                        unsigned int outside = 0;
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if ((left >> (o0 + k * P) & ((1u << P) - 1u)) != 0) {
                                const int o = o0 + k * P + sub;  // the lane whose half it is
                                at[k] = ((x & 1) ? o ^ 16 : o) * M + (o >> 4) * MH + m;
                                const int g = left >> o & 1u ? base[at[k]] : wb;
                                v[k] = __int_as_float(0x7fc00000);
                                if ((unsigned int)(g - wb) >= (unsigned int)wn) {
                                    outside |= 1u << k;
                                    if ((unsigned int)g < (unsigned int)(E * N))
                                        v[k] = __ldg(a.u + g);
                                    else
                                        atomicOr(a.err, 2u);
                                }
                            }
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (outside >> k & 1u)
                                base[at[k]] = __float_as_int(v[k]);
                    }
                    __syncwarp();
                }
            } else if (__any_sync(0xffffffffu, far >= (unsigned int)wn)) {
                parked = true;
                if (live) {
                    // eight at a time: their loads are in flight together
                    for (int mb = 0; mb < MH; mb += 8) {
                        float v[8];
                        unsigned int outside = 0;
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const int g = mb + k < MH && m0 + mb + k < M ? vr[mb + k] : wb;
                            v[k] = __int_as_float(0x7fc00000);
                            if ((unsigned int)(g - wb) >= (unsigned int)wn) {
                                outside |= 1u << k;
                                if ((unsigned int)g < (unsigned int)(E * N))
                                    v[k] = __ldg(a.u + g);
                                else
                                    atomicOr(a.err, 2u);
                            }
                        }
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (outside >> k & 1u)
                                vr[mb + k] = __float_as_int(v[k]);
                    }
                }
                __syncwarp();
            }
            const uint32_t own = win_s + (uint32_t)((e0 - lo + warp * CH + rr) * N) * 4u, park = smem_addr(vr);
            float f[MH];
#pragma unroll
            for (int m = 0; m < MH; m += 4) {
                const int4 node = *reinterpret_cast<const int4 *>(fnode + m0 + m);
                const int nd[4] = {node.x, node.y, node.z, node.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t ext = (unsigned int)q[m + k] < (unsigned int)wn ? win_s + 4u * (uint32_t)q[m + k]
                                                                                   : park + 4u * (m + k);
                    f[m + k] = __fsub_rn(lds_f32(own + nd[k]), lds_f32(ext));
                }
            }
#pragma unroll
            for (int m = 0; m < MH; ++m) {
                // the scale of face m0 + m (no branches: they would hold up the loads around them)
                const float sc = m >= b1 ? (m >= b2 ? (m >= b3 ? sv[3] : sv[2]) : sv[1]) : sv[0];
                f[m] = m < MH - 8 || m0 + m < M ? __fmul_rn(sc, f[m]) : 0.f;
                seen |= __float_as_uint(f[m]);
            }
#pragma unroll
            for (int m = 0; m < MH; m += 2)
                fx[x][m / 2] = pack_f32x2(f[m], f[m + 1]);
        }
        if (!ok) {
            if (lane == 0)
                atomicOr(a.err, 1u);
            break;
        }
        // Every load of the window and of A must have returned before they are handed to the next
        // bulk copies: the branch depends on all the values, what follows on the branch.
        if (seen == 0x7fb5a5a5u)
            __nanosleep(0);
        if (parked)
            fence_async_smem();
        __threadfence_block();
        __syncwarp();
        if (nt < ntiles) {
            scales(nt);
            if (lane == 0) {
                fetch(nt, vA, abar, 0, 32);
                if ((atomicAdd(gathered, 1u) + 1u) % (unsigned int)W == 0) {
                    __threadfence_block();
                    window(nt);
                }
            }
        }
        float *o0 = stage + lane * N;
        for (int i = 0; i < N; i += 4) {
            float r[EPT][4];
            row_columns<MH, EPT, 2 * MH>(Ls + (size_t)i * 2 * MH + m0, fx, r);
#pragma unroll
            for (int x = 0; x < EPT; x += 2) {
                float *o = o0 + 16 * x * N + i;
                float v[4];
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    v[m] = r[x][m] + __shfl_xor_sync(0xffffffffu, r[x + 1][m], 16);
                if ((N & 3) == 0) {
                    *reinterpret_cast<float4 *>(o) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int m = 0; m < 4; ++m)
                        if (i + m < N)
                            o[m] = v[m];
                }
            }
        }
        const int total = rows * N;
        float *dst = a.out + ((long long)e0 + warp * CH) * N;
        fence_async_smem();
        __syncwarp();
        if (!a.accumulate && a.bulk_store && (total & 3) == 0) {
            if (lane == 0) {
                bulk_s2g(dst, stage, (uint32_t)total * 4u);
                bulk_commit();
                bulk_wait_read0();
            }
        } else if (a.bulk_store && (total & 3) == 0) {
            float4 *d4 = reinterpret_cast<float4 *>(dst);
            const float4 *s4 = reinterpret_cast<const float4 *>(stage);
#pragma unroll 4
            for (int k = lane; k < total / 4; k += 32) {
                float4 o = d4[k];
                const float4 v = s4[k];
                o.x = __fadd_rn(o.x, v.x), o.y = __fadd_rn(o.y, v.y);
                o.z = __fadd_rn(o.z, v.z), o.w = __fadd_rn(o.w, v.w);
                d4[k] = o;
            }
            fence_async_smem();  // a bulk copy may write the staging buffer next
        } else {
            for (int k = lane; k < total; k += 32)
                dst[k] = a.accumulate ? __fadd_rn(dst[k], stage[k]) : stage[k];
            fence_async_smem();
        }
        __syncwarp();
        if (lane == 0 && nt < ntiles)
            fetch(nt, vB, bbar, 32, CH - 32);
    }
    if (lane == 0)
        bulk_wait0();
}

template <int MH, bool LINES = false>
static void *lift_row_of(int ept)
{
    return ept == 2 ? reinterpret_cast<void *>(&lift_row_kernel<MH, 2, LINES>)
                    : reinterpret_cast<void *>(&lift_row_kernel<MH, lift_row_ept(MH), LINES>);
}

static void *lift_row_fn(int mh, int ept, bool lines)
{
    switch (mh) {
    case 4: return lift_row_of<4>(ept);
    case 8: return lift_row_of<8>(ept);
    case 12: return lift_row_of<12>(ept);
    case 16: return lines ? lift_row_of<16, true>(ept) : lift_row_of<16>(ept);
    case 20: return lift_row_of<20>(ept);
    case 24: return lift_row_of<24>(ept);
    case 28: return lift_row_of<28>(ept);
    case 32: return lines ? lift_row_of<32, true>(ept) : lift_row_of<32>(ept);
    default: return nullptr;
    }
}

// Which of the two kernels is the faster one, measured over N = 8 to 128 and M = 12 to 64 with
// neighbours up to 64 elements away (us, tiled -> rows in registers).  Rows of 32 or 64 values meet
// in one bank (N = 64, M = 64, E = 300007: 110 -> 167).  Long rows leave few warps beside the window
// (N = 50, M = 30: 66 -> 84; N = 40, M = 60: 92 -> 74, but N = 37 104 -> 121 with neighbours 200 away); a
// batch of one or a few warps an SM waits for those warps' products (E = 4099: N = 27, M = 27 5.9 ->
// 6.3, N = 35, M = 60 8.8 -> 7.9; E = 12000: N = 60, M = 60 12.6 -> 11.0).  Accumulating, the tiled
// kernel's reads of out weigh more than all that (N = 60, M = 60, E = 300007: 231 -> 142), and in small
// batches more than the bank conflicts of N = 32 (M = 60, E = 14000: 13.0 -> 10.2; N = 64 14.3 -> 13.4,
// but E = 9000 11.5 -> 12.2).
static bool lift_row_faster(long long E, int N, int M, bool accumulate, int sms)
{
    const long long per_sm = E / sms;
    if (N % 32 == 0)
        return N == 32 && accumulate && per_sm < 96;
    if (accumulate)
        return true;
    if (M >= 40)
        return N <= (per_sm < 32 ? 40 : per_sm < 96 ? 63 : per_sm < 512 ? 45 : 36);
    return N <= (per_sm < 32 ? 24 : 36);
}

// Warps with a chunk each (the others only help to lay out L): the number that ends soonest, a tile
// costing about its chunks and two more for what does not depend on them.  Scales are staged unless
// that costs a warp.
LiftRowPlan lift_row_plan(long long E, int N, int M, int Nf, bool accumulate, int sms, size_t cap)
{
    LiftRowPlan p{};
    if (Nf > 4 || M > kLiftRowMaxM || E < 1 || E >= 1ll << 30)  // (tile bounds are ints)
        return p;
    if (!lift_row_faster(E, N, M, accumulate, sms))
        return p;
    p.ept = E <= 96ll * sms ? 2 : lift_row_ept(lift_row_half(M));
    const int ch = 16 * p.ept;
    const long long chunks = (E + ch - 1) / ch;
    p.halo = 64;
    long long best = 0;
    int most = 0;
    for (int w = kLiftRowWarps; w >= 1; --w)
        for (int stage_s = 1; stage_s >= 0; --stage_s) {
            const size_t smem = lift_row_smem(N, M, Nf, p.ept, w, p.halo, stage_s).total;
            if (smem > cap)
                continue;
            most = std::max(most, w);
            const long long tiles = (chunks + w - 1) / w, cost = (tiles + sms - 1) / sms * (w + 2);
            if (p.warps == 0 || cost < best) {
                best = cost;
                p.warps = w;
                p.stage_s = stage_s;
                p.smem = smem;
                p.tiles = tiles;
            }
            break;
        }
    if (most < 4 && chunks > (long long)most * sms)
        p.warps = 0;  // long rows of u: too few warps fit beside one window
    // few tiles: a far trace's latency weighs more than reading more of u from L2 (degree 4, E = 100003,
    // neighbours 200 elements away: 46 -> 31 us; E = 50000, 64 away: 17.3 -> 17.9)
    while (p.warps > 0 && p.tiles <= 2ll * sms && p.halo < 256) {
        const size_t smem = lift_row_smem(N, M, Nf, p.ept, p.warps, p.halo + 32, p.stage_s).total;
        if (smem > cap)
            break;
        p.smem = smem;
        p.halo += 32;
    }
    return p;
}

lc_status lift_row_launch(const LiftArgs &a, int ept, int grid, size_t smem, cudaStream_t s)
{
    void *fn = lift_row_fn(lift_row_half(a.M), ept, a.M % 32 == 0);
    if (!fn)
        return LC_ERR_INVALID_VARIANT;
    cudaError_t e = allow_smem(fn);
    if (e != cudaSuccess)
        return cuda_fail(e);
    LiftArgs args = a;
    void *params[] = {&args};
    e = cudaLaunchKernel(fn, dim3(grid), dim3(32 * kLiftRowWarps), params, smem, s);
    return e == cudaSuccess ? LC_OK : cuda_fail(e);
}

}  // namespace lc
