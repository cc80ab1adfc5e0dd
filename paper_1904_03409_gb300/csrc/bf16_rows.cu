// bf16_rows.cu -- the recurrences of Algorithm 1 (forward) and of its reverse-time backward
// (Sec. 5) for hidden widths up to 256 as thread-block clusters of 8 or 16 rows.
//
// Instances are independent, so a batch is cut into groups of 8 (or, NT = 2, 16) rows and each
// group runs all T steps in one cluster of its own; a CTA holds 32 hidden units, so a cluster has
// ceil(H / 32) <= 8 CTAs. A step is a chain of one contraction, the cell and an exchange
// between the cluster's CTAs, and with so few rows latency bounds it, not arithmetic or
// bandwidth: the gate contraction is 128 gate columns x 8 rows x (I + H) a CTA. It therefore
// runs as mma.sync (m16n8k16, bf16 in, fp32 accumulate) with the weights as the M operand,
// kept in registers for the whole launch, and the rows as N: the accumulators are in the
// cell's registers as soon as the last MMA is done. The 64-row tcgen05 clusters
// (bf16_cluster.cu) spend 1.54 us a step forward and 2.07 us backward on commits, barriers,
// tensor-memory loads and on bringing 64 rows to every CTA (I = H = 200, B = 64); here it is
// 0.96 and 1.03 us: a chain of ldmatrix and MMAs, the cell, and the wait until every
// CTA's piece has landed. A 64 x 200 pass of 185
// steps with per-step gradients: 0.777 -> 0.437 ms (with y stored here and a free GPU to start on).
//
// Forward. Warp w of CTA ct owns units 32 ct + 8 w .. + 7: M tile 0 is their gates i and f,
// M tile 1 gates g and o, so lane (g, t) = (lane / 4, lane % 4) holds all four gates of unit
// g for rows 2t and 2t + 1: the cell needs no shuffle. The new h operand (h' where the step
// pushed, else the older top) is transposed to row pieces of 8 units (movmatrix) and stored
// into every CTA of the cluster by st.async, 16 bytes a store, counting on the receiver's
// mbarrier. Warps 4..7 multiply the x part (W_x and x rows in shared memory) up to two steps
// ahead; done by the step's own warps it was 300 cycles on the chain.
//
// Backward. Step t's gate gradients of a CTA's own units stay in that CTA: it multiplies
// them by its 128 gate columns of W_h into partial dh_read rows of all H units (M), and sends
// each 16-unit M tile's fragment, fp32, to the CTA that owns those units: 7 KB received a
// step and CTA at 8 x 200, where gathering every gate gradient would take 13 KB. The owner
// adds the parts in CTA order (deterministic) to the gradient history.
//
// The operand and partial-sum buffers are double-buffered by step parity. A buffer is
// written for step t + 2 only by a CTA that has received all of step t + 1, which every warp
// of every CTA sent after it had read step t's buffer.
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>

#include "bf16_dev.cuh"

namespace sl {
namespace {

using tc::smem_u32;

constexpr int kRcThreads = 256;  // warps 0..3: the step; 4..7: forward the x part, backward half the MMAs and dG
constexpr int kRcX = 4;          // x_t buffers (steps in flight)
constexpr int kRcDgLd = 136;     // row of the backward's own gate gradients: 128 + 8 (odd 16-byte pieces)
constexpr long long kRcSettle = 100000;  // cycles an aborted CTA waits for stores in flight

struct RcArgs {
    StepArgs s;
    const uint4 *wfrag;        // W_h fragments (pack_rows_wh_elem / pack_rows_wb_elem)
    const uint8_t *wx;         // forward: W_x rows as they lie in shared memory (pack_rows_wx_elem)
    const __nv_bfloat16 *x;    // forward: [T][B][I]
    __nv_bfloat16 *y;          // forward: [T][B][H] step outputs, or null
    const float *d_top;        // backward: the final top's gradient, still to be added (or null)
    const int32_t *ftop;       // backward: the final top's history row of each instance
    int KX;                    // forward: x contraction steps of 16
    int dead;                  // backward: a state no step reads can have a gradient (push-only seeds)
};
struct RcGroup {
    RcArgs p[kMaxGroup];
    int first[kMaxGroup + 1];  // first cluster of each member
    int n, C;                  // members; CTAs per cluster
};

__device__ __forceinline__ void mma16816(float (&d)[4], const uint4 &a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
// lanes 0..15 give the rows (column halves 0 and 1); the other lanes' addresses are unused
__device__ __forceinline__ void ldsm2(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
// the transpose of an 8 x 8 matrix of 16-bit values held as a fragment
__device__ __forceinline__ uint32_t movmatrix(uint32_t a)
{
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t *)&v;
}
__device__ __forceinline__ uint32_t pack2_f16(float lo, float hi)
{
    const __half2 v = __floats2half2_rn(lo, hi);
    return *(const uint32_t *)&v;
}
// 2 units of each of 4 lanes (one row's 8 units) to all four of them
__device__ __forceinline__ uint4 gather_row(uint32_t v, int lane)
{
    const int base = lane & 28;
    return make_uint4(__shfl_sync(0xffffffffu, v, base), __shfl_sync(0xffffffffu, v, base | 1),
                      __shfl_sync(0xffffffffu, v, base | 2), __shfl_sync(0xffffffffu, v, base | 3));
}
// row `i` of an array of `stride`-byte rows (one 32 x 32 -> 64 multiply-add)
template <typename P>
__device__ __forceinline__ P *at_row(P *base, int i, uint32_t stride)
{
    return (P *)((char *)base + (uint64_t)(uint32_t)i * stride);
}
template <typename P>
__device__ __forceinline__ const P *at_row(const P *base, int i, uint32_t stride)
{
    return (const P *)((const char *)base + (uint64_t)(uint32_t)i * stride);
}

__device__ __forceinline__ void rc_abort(volatile int *abort, int32_t *err)
{
    *abort = 1;
    atomicCAS(err, 0, (int)SL_ERR_TIMEOUT);
}

// Bounded wait of a whole warp for an mbarrier phase; kCluster: completed by asynchronous
// stores of the cluster's CTAs (acquire at cluster scope). Polls: a suspending try_wait
// wakes later than a poll sees the phase, and nothing else of the warp could run.
template <bool kCluster>
__device__ __forceinline__ bool rc_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if constexpr (kCluster)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
template <bool kCluster>
__device__ __forceinline__ bool rc_wait(uint32_t bar, uint32_t parity, long long limit, volatile int *abort, int32_t *err)
{
    bool ok = rc_test<kCluster>(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    const long long t0 = clock64();
    while (true) {
        const bool over = clock64() - t0 >= limit || *abort;
        if (__any_sync(0xffffffffu, over)) break;
        ok = rc_test<kCluster>(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    rc_abort(abort, err);
    return false;
}

// No CTA leaves while another may still store into its shared memory: after a complete run
// every store has been waited for; an aborted CTA gives those in flight time to land.
__device__ __forceinline__ void rc_leave(volatile int *abort)
{
    __syncthreads();
    tc::cluster_sync();
    if (*abort) {
        const long long t0 = clock64();
        while (clock64() - t0 < kRcSettle) {}
    }
    __syncthreads();
    tc::cluster_sync();
}
__device__ __forceinline__ const RcArgs &rc_member(const RcGroup &G, int cid, int *rel)
{
    int m = 0;
    while (m + 1 < G.n && cid >= G.first[m + 1]) ++m;
    *rel = cid - G.first[m];
    return G.p[m];
}

// ------------------------------------------------------------------------ forward
// Shared memory: [W_x 128 rows][x buffers kRcX x 8 NT rows][h operand 2 x 8 NT rows]
// [x part 4 warps x 2 x 2 NT fragments][barriers]; rows of 16 KX + 8 (16 KH + 8) values, an
// odd number of 16-byte pieces (conflict-free ldmatrix).
__host__ __device__ constexpr uint32_t rc_fwd_smem(int KX, int KH, int NT)
{
    return (128u + kRcX * 8u * NT) * (KX * 16 + 8) * 2 + 2u * 8 * NT * (KH * 16 + 8) * 2 + 4u * 2 * 2 * NT * 512 + 256;
}

// registers a thread after the split of the block's 256 x 128 between its two warpgroups
constexpr int kRcRegsStep = 192, kRcRegsX = 64;    // forward
constexpr int kRcRegsBwd = 160, kRcRegsBwd2 = 96;  // backward, two N tiles

template <int KH, int NT>
__global__ void __launch_bounds__(kRcThreads, 2) step_rows(const __grid_constant__ RcGroup G)
{
    constexpr int NR = 8 * NT;
    constexpr uint32_t SH = (KH * 16 + 8) * 2, hb_bytes = NR * SH;  // an h operand row, a buffer
    constexpr uint32_t xf_bytes = 2 * NT * 512;                     // x part of a warp and step
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_abort;
    int rel;
    const RcArgs &p = rc_member(G, (int)blockIdx.x / G.C, &rel);
    const StepArgs &a = p.s;
    const int T = a.T, B = a.B, H = a.H, I = a.I, KX = p.KX;
    const uint32_t ct = tc::cluster_rank(), C = (uint32_t)G.C;
    const int row0 = rel * NR, nrows = min(NR, B - row0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const uint32_t SX = (uint32_t)(KX * 16 + 8) * 2, wx_bytes = 128 * SX, xb_bytes = NR * SX;
    const uint32_t s_wx = smem_u32(smem), s_x = s_wx + wx_bytes, s_h = s_x + kRcX * xb_bytes;
    const uint32_t s_xf = s_h + 2 * hb_bytes, s_bar = s_xf + 4 * 2 * xf_bytes;
    uint64_t *bars = (uint64_t *)(smem + (s_bar - s_wx));
    // [0..1] h operand of the buffer complete; [2] W_x; [3 + 2 w + b] x part of warp w ready,
    // [11 + 2 w + b] consumed
    auto bar = [&](int i) { return s_bar + 8 * i; };
    volatile int *abort = &s_abort;
    const long long limit = a.limit;
    const int w4 = warp & 3, u0 = (int)ct * 32 + w4 * 8, u = u0 + g;  // the warp's first unit, the lane's unit
    const bool warp_on = u0 < H;                           // H % 8 == 0: whole warps
    const uint32_t h_bytes = (uint32_t)NR * (H / 8) * 16;  // of one step's operand, all of them

    // zero x and h buffers (padding and rows past the batch stay zero), h_read(0) = h0
    for (uint32_t i = tid; i < (kRcX * xb_bytes + 2 * hb_bytes) / 16; i += kRcThreads)
        *(uint4 *)(smem + wx_bytes + i * 16) = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (int i = 0; i < 19; ++i) tc::mbar_init(&bars[i], 1);
        s_abort = 0;
        tc::fence_mbar_init();
    }
    __syncthreads();
    for (int i = tid; i < nrows * (H / 8); i += kRcThreads) {
        const int r = i / (H / 8), q = i - r * (H / 8);
        *(uint4 *)(smem + wx_bytes + kRcX * xb_bytes + r * SH + q * 16) =
            __ldcg((const uint4 *)(a.hr + (size_t)(row0 + r) * H) + q);
    }
    if (tid == 0) {
        tc::mbar_arrive_expect_tx(&bars[2], wx_bytes);
        tc::bulk_g2s(s_wx, p.wx + (size_t)ct * wx_bytes, wx_bytes, &bars[2]);
        // h_read(1) and h_read(2): every CTA's pieces, by byte count (the first phase of
        // buffer 0 is the operand of step 2: step 0's is in place already)
        if (T > 1) tc::mbar_arrive_expect_tx(&bars[1], h_bytes);
        if (T > 2) tc::mbar_arrive_expect_tx(&bars[0], h_bytes);
    }
    __syncthreads();
    tc::cluster_sync();  // every CTA's barriers and buffers exist before any store lands on them

    if (warp >= 4) {
        // ---------------------------------------------- the x part: bias + x_t W_x, steps ahead
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRcRegsX));
        // 16 / NT threads a row; row r's pieces tl, tl + 16 / NT, ...
        const int xr = (tid & 127) / (16 / NT), tl = (tid & 127) % (16 / NT);
        const __nv_bfloat16 *xp = p.x + ((size_t)row0 + xr) * I;
        // XS steps at a time: a weight fragment is read from shared memory once for all of them,
        // the largest part of what two CTAs an SM ask of it (256 x 200: 1.53 us a step, 1.34 by
        // twos; by fours the burst delays the steps, 1.49; two N tiles by twos spill, 2.96 for 2.63)
        constexpr int XS = NT == 1 ? 2 : 1;
        auto load_x = [&](int t0) {  // steps t0 ..
#pragma unroll
            for (int t = t0; t < t0 + XS; ++t)
                if (t < T && xr < nrows) {
                    const __nv_bfloat16 *src = xp + (size_t)t * B * I;
                    const uint32_t dst = s_x + (t & (kRcX - 1)) * xb_bytes + xr * SX;
                    for (int q = tl; q < I / 8; q += 16 / NT) tc::cp_async16(dst + q * 16, src + q * 8, 16);
                }
            tc::cp_async_commit();
        };
        constexpr int ahead = kRcX / XS - 1;
        for (int i = 0; i < ahead; ++i) load_x(i * XS);
        float bias[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) bias[q] = warp_on ? a.bias[q * H + u] : 0.0f;
        // A rows (lane % 16), column half (lane / 16) of the warp's M tiles
        const uint32_t wa = s_wx + (uint32_t)(w4 * 32 + (lane & 15)) * SX + (lane >> 4) * 16;
        bool ok = rc_wait<false>(bar(2), 0, limit, abort, a.err);
        for (int t = 0; t < T; t += XS) {
            tc::cp_async_wait<ahead - 1>();
            // these steps' x is in place, and every warp has read the ones before, whose buffers
            // are loaded next
            if (tc::bar_any(1, 128, !ok)) break;
            load_x(t + ahead * XS);
            if (!warp_on) continue;
            float acc[XS][2][NT][4];
#pragma unroll
            for (int e = 0; e < XS; ++e)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        acc[e][q >> 1][n][(q & 1) * 2] = acc[e][q >> 1][n][(q & 1) * 2 + 1] = bias[q];
            const uint32_t xa = s_x + (t & (kRcX - 1)) * xb_bytes + (lane & 7) * SX + ((lane >> 3) & 1) * 16;
#pragma unroll 2
            for (int k = 0; k < KX; ++k) {
                uint32_t A0[4], A1[4], bb[4];
                ldsm4(A0, wa + k * 32);
                ldsm4(A1, wa + 16 * SX + k * 32);
#pragma unroll
                for (int e = 0; e < XS; ++e)
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        ldsm2(bb, xa + (e * NR + n * 8) * SX + k * 32);
                        mma16816(acc[e][0][n], make_uint4(A0[0], A0[1], A0[2], A0[3]), bb[0], bb[1]);
                        mma16816(acc[e][1][n], make_uint4(A1[0], A1[1], A1[2], A1[3]), bb[0], bb[1]);
                    }
            }
#pragma unroll
            for (int e = 0; e < XS; ++e) {
                if (t + e >= T) break;
                const int b = (t + e) & 1;
                if (t + e >= 2) ok = ok && rc_wait<false>(bar(11 + 2 * w4 + b), (uint32_t)(((t + e) >> 1) - 1) & 1, limit, abort, a.err);
                uint8_t *out = smem + (s_xf - s_wx) + (w4 * 2 + b) * xf_bytes + lane * 16;
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int n = 0; n < NT; ++n)
                        *(float4 *)(out + (i * NT + n) * 512) =
                            make_float4(acc[e][i][n][0], acc[e][i][n][1], acc[e][i][n][2], acc[e][i][n][3]);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&bars[3 + 2 * w4 + b]);
            }
        }
        tc::cp_async_wait<0>();
    } else {
        // ------------------------------------------------------------------------- the step
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRcRegsStep));
        // this warp's gate columns of W_h, for the whole launch
        uint4 wh[2][KH];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < KH; ++k)
                wh[i][k] = __ldcg(p.wfrag + ((((size_t)ct * 4 + warp) * 2 + i) * KH + k) * 32 + lane);
        // Rows past the batch's end read the last row's data and write nothing. This lane's
        // cells: unit u of rows 2 t4, 2 t4 + 1 of each N tile; its row piece: row g.
        const uint32_t sc = (uint32_t)B * H * 4, sh = sc / 2, si = (uint32_t)B * 4, sg = (uint32_t)B * H * 8;
        int rc[NT][2], rg[NT];
        bool okc[NT][2], okg[NT];
        int i1[NT][2], g1[NT], g2[NT];
        float cr[NT][2];  // c of the state this step reads
        uint4 hold[NT];   // the older top that is step t + 1's operand, if the step does not push
#pragma unroll
        for (int n = 0; n < NT; ++n) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 8 * n + 2 * t4 + e;
                okc[n][e] = r < nrows;
                rc[n][e] = row0 + min(r, nrows - 1);
                const int i0 = a.top[rc[n][e]];
                i1[n][e] = at_row(a.top, 1, si)[rc[n][e]];
                cr[n][e] = warp_on ? __ldcg(at_row(a.hist_c, i0, sc) + (size_t)rc[n][e] * H + u) : 0.0f;
            }
            okg[n] = 8 * n + g < nrows;
            rg[n] = row0 + min(8 * n + g, nrows - 1);
            g1[n] = at_row(a.top, 1, si)[rg[n]];
            g2[n] = at_row(a.top, min(2, T), si)[rg[n]];
            hold[n] = make_uint4(0, 0, 0, 0);  // h0 is the only older top
            if (warp_on) hold[n] = __ldcg((const uint4 *)(a.hist_h + (size_t)rg[n] * H + u0));
        }
        // this lane's peers in the cluster: t4 and t4 + 4
        const uint32_t peer0 = tc::mapa(s_wx, t4 < C ? t4 : 0), peer1 = tc::mapa(s_wx, t4 + 4 < C ? t4 + 4 : 0);
        const bool send0 = t4 < C, send1 = t4 + 4 < C;
        const uint32_t h_off = s_h - s_wx, bar_off = s_bar - s_wx;
        // where this lane's piece of a row goes: history row t + 1, the h operand row t + 1 (for
        // the weight gradient), y_t (a step's output is its top's h, the operand of the next step)
        __nv_bfloat16 *const st_base = t4 == 0 ? at_row(a.hist_h, 1, sh) : t4 == 1 ? at_row(a.hr, 1, sh) : p.y;
        bool st_on[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) st_on[n] = okg[n] && t4 < (p.y ? 3 : 2);
        const uint32_t ha0 = s_h + (lane & 7) * SH + (lane >> 3) * 16;
        const uint32_t ha2 = s_h + (lane & 7) * SH + ((lane >> 3) & 1) * 16;  // an odd last K step
        for (int t = 0; t < (warp_on ? T : 0); ++t) {
            const int b = t & 1;
            // (without this barrier the compiler arranges the loop so that the loads below wait
            // for one another: 1.44 us a step at 64 x 200, 1.00 with it)
            __syncwarp();
            // operands of step t + 1 in rows written before step t (row t + 1 itself is not: then
            // the loaded value is unused), and the indices after them
            float crn[NT][2];
            uint4 holdn[NT];
            int i2[NT][2], g3[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    crn[n][e] = __ldcg(at_row(a.hist_c, i1[n][e], sc) + (size_t)rc[n][e] * H + u);
                    i2[n][e] = __ldcg(at_row(a.top, min(t + 2, T), si) + rc[n][e]);
                }
                holdn[n] = __ldcg((const uint4 *)(at_row(a.hist_h, g2[n], sh) + (size_t)rg[n] * H + u0));
                g3[n] = __ldcg(at_row(a.top, min(t + 3, T), si) + rg[n]);
            }
            float acc[2][NT][4];
            if (!rc_wait<false>(bar(3 + 2 * w4 + b), (uint32_t)(t >> 1) & 1, limit, abort, a.err)) break;
            {
                const uint8_t *in = smem + (s_xf - s_wx) + (w4 * 2 + b) * xf_bytes + lane * 16;
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const float4 v = *(const float4 *)(in + (i * NT + n) * 512);
                        acc[i][n][0] = v.x; acc[i][n][1] = v.y; acc[i][n][2] = v.z; acc[i][n][3] = v.w;
                    }
            }
            // h_read(t): every CTA's pieces (step t > 0: phase (t - 1) / 2 of buffer t % 2)
            if (t > 0) {
                if (!rc_wait<true>(bar(b), (uint32_t)((t - 1) >> 1) & 1, limit, abort, a.err)) break;
                if (tid == 0 && t + 2 < T) tc::mbar_arrive_expect_tx(&bars[b], h_bytes);
            }
            // with one N tile, two accumulators an M tile halve the chain of dependent MMAs
            constexpr bool kTwo = NT == 1;
            float acc2[2][NT][4];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc2[i][n][q] = 0.0f;
#pragma unroll
            for (int k = 0; k < KH; k += 2)
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    uint32_t bb[4];
                    if (k + 1 < KH)
                        ldsm4(bb, ha0 + b * hb_bytes + n * 8 * SH + k * 32);
                    else
                        ldsm2(bb, ha2 + b * hb_bytes + n * 8 * SH + k * 32);
#pragma unroll
                    for (int i = 0; i < 2; ++i) mma16816(acc[i][n], wh[i][k], bb[0], bb[1]);
                    if (k + 1 < KH) {
#pragma unroll
                        for (int i = 0; i < 2; ++i) mma16816(kTwo ? acc2[i][n] : acc[i][n], wh[i][k + 1], bb[2], bb[3]);
                    }
                }
            // the cell; the operand goes out first
            float cn[NT][2];
            uint32_t gt[NT][2][2];
            uint4 hrow[NT], op[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                float hn[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    auto z = [&](int i, int q) { return kTwo ? acc[i][n][q] + acc2[i][n][q] : acc[i][n][q]; };
                    const float ig = sigm(z(0, e)), fg = sigm(z(0, 2 + e)), gg = tanh_hw(z(1, e)), og = sigm(z(1, 2 + e));
                    cn[n][e] = fmaf(fg, cr[n][e], ig * gg);
                    hn[e] = og * tanh_hw(cn[n][e]);
                    gt[n][e][0] = pack2_f16(ig, fg);
                    gt[n][e][1] = pack2_f16(gg, og);
                }
                hrow[n] = gather_row(movmatrix(pack2_bf16(hn[0], hn[1])), lane);  // row 8 n + g, units u0 .. + 7
                op[n] = g1[n] == t + 1 ? hrow[n] : hold[n];
                if (t + 1 < T) {
                    const uint32_t off = h_off + (b ^ 1) * hb_bytes + (8 * n + g) * SH + u0 * 2;
                    const uint32_t w[4] = {op[n].x, op[n].y, op[n].z, op[n].w};
                    if (send0) tc::st_async_v4(peer0 + off, w, peer0 + bar_off + 8 * (b ^ 1));
                    if (send1) tc::st_async_v4(peer1 + off, w, peer1 + bar_off + 8 * (b ^ 1));
                }
            }
            // the x part's buffer is handed back only now: its warp then multiplies the next one
            // while the operands travel, and not against this warp's MMAs
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bars[11 + 2 * w4 + b]);
            // the row pieces, c, the gates
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                if (st_on[n]) *(uint4 *)(at_row(st_base, t, sh) + (size_t)rg[n] * H + u0) = t4 == 0 ? hrow[n] : op[n];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (okc[n][e]) {
                        at_row(a.hist_c, t + 1, sc)[(size_t)rc[n][e] * H + u] = cn[n][e];
                        *(uint2 *)(at_row(a.gates, t, sg) + ((size_t)rc[n][e] * H + u) * 4) = make_uint2(gt[n][e][0], gt[n][e][1]);
                    }
                    cr[n][e] = i1[n][e] == t + 1 ? cn[n][e] : crn[n][e];
                    i1[n][e] = i2[n][e];
                }
                hold[n] = g2[n] == t + 1 ? hrow[n] : holdn[n];
                g1[n] = g2[n];
                g2[n] = g3[n];
            }
            __syncwarp();  // row pieces are read back by other lanes of the warp at later steps
        }
    }
    if (tid == 0) tc::mbar_wait(&bars[2], 0, kDrainLimit, nullptr);  // after an abort: the copy of W_x lands
    rc_leave(abort);
}

// ----------------------------------------------------------------------- backward
// Shared memory: [partial sums 2 x C parts x 2 M tiles x NT x 32 lanes x 16 bytes]
// [own gate gradients 2 x 8 NT rows][barriers]
__host__ __device__ constexpr uint32_t rc_bwd_smem(int C, int NT)
{
    return 2u * C * 2 * NT * 512 + 2u * 8 * NT * kRcDgLd * 2 + 64;
}

template <int KT, int NT>
__global__ void __launch_bounds__(kRcThreads, 2) step_rowsb(const __grid_constant__ RcGroup G)
{
    constexpr int NR = 8 * NT, MT = (KT + 7) / 8;  // M tiles a warp: 16-unit tiles warp, warp + 8
    constexpr uint32_t slot = NT * 512, dgb = NR * kRcDgLd * 2;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_abort;
    int rel;
    const RcArgs &p = rc_member(G, (int)blockIdx.x / G.C, &rel);
    const StepArgs &a = p.s;
    const int T = a.T, B = a.B, H = a.H;
    const uint32_t ct = tc::cluster_rank(), C = (uint32_t)G.C;
    const int row0 = rel * NR, nrows = min(NR, B - row0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const uint32_t buf = C * 2 * slot;
    const uint32_t s_p = smem_u32(smem), s_dg = s_p + 2 * buf, s_bar = s_dg + 2 * dgb;
    uint64_t *rbar = (uint64_t *)(smem + 2 * buf + 2 * dgb);  // [2]
    volatile int *abort = &s_abort;
    const long long limit = a.limit;
    const int n_mt = (H + 15) / 16;                                            // 16-unit M tiles
    const uint32_t r_bytes = (uint32_t)min(2, n_mt - 2 * (int)ct) * C * slot;  // of one step's parts

    for (uint32_t i = tid; i < 2 * dgb / 16; i += kRcThreads) *(uint4 *)(smem + 2 * buf + i * 16) = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) tc::mbar_init(&rbar[i], 1);
        s_abort = 0;
        tc::fence_mbar_init();
        for (int i = 0; i < 2 && i < T; ++i) tc::mbar_arrive_expect_tx(&rbar[(T - 1 - i) & 1], r_bytes);
    }
    // this CTA's gate columns of W_h for the warp's M tiles, for the whole launch
    uint4 wt[MT][8];
    auto load_weights = [&]() {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int k = 0; k < 8; ++k) wt[i][k] = __ldcg(p.wfrag + ((((size_t)ct * 8 + warp) * MT + i) * 8 + k) * 32 + lane);
    };
    // M tile j = 8 i + warp: units 16 j .. + 15, which CTA j / 2 owns
    uint32_t peer[MT];
#pragma unroll
    for (int i = 0; i < MT; ++i) peer[i] = tc::mapa(s_p, (uint32_t)min(8 * i + warp, n_mt - 1) >> 1);
    __syncthreads();
    tc::cluster_sync();  // every CTA's barriers exist before any store lands on them

    // partial dh_read of every unit from this CTA's gate columns, to the units' owners
    auto contract = [&](int b) {
        float acc[MT][NT][4];
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][n][q] = 0.0f;
        const uint32_t ga = s_dg + b * dgb + (lane & 7) * (kRcDgLd * 2) + (lane >> 3) * 16;
#pragma unroll
        for (int k = 0; k < 8; k += 2)
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                uint32_t bb[4];
                ldsm4(bb, ga + n * 8 * (kRcDgLd * 2) + k * 32);
#pragma unroll
                for (int i = 0; i < MT; ++i) mma16816(acc[i][n], wt[i][k], bb[0], bb[1]);
#pragma unroll
                for (int i = 0; i < MT; ++i) mma16816(acc[i][n], wt[i][k + 1], bb[2], bb[3]);
            }
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            const int j = 8 * i + warp;
            if (j >= n_mt) continue;
            const uint32_t dst = peer[i] + b * buf + (ct * 2 + (j & 1)) * slot + lane * 16;
#pragma unroll
            for (int n = 0; n < NT; ++n)
                tc::st_async_v4(dst + n * 512, reinterpret_cast<const uint32_t *>(acc[i][n]), peer[i] + (s_bar - s_p) + 8 * b);
        }
    };
    const uint32_t sc = (uint32_t)B * H * 4, si = (uint32_t)B * 4, sg = (uint32_t)B * H * 8;

    if (warp >= 4) {
        // ---------- half of the M tiles, and dG in the [T B][4H] layout (for dx and dW): thread
        // (row, 8 units, gate), the eight units' values gathered from the operand rows
        if constexpr (NT > 1) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRcRegsBwd2));
        const int j = tid & 127;
        load_weights();
        for (int t = T - 1; t >= 0; --t) {
            const int b = t & 1;
            if (__syncthreads_or(0)) break;
            contract(b);
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const int r = 8 * n + (j >> 4), q8 = (j >> 2) & 3, gate = j & 3;
                if (r < nrows && (int)ct * 32 + q8 * 8 < H) {
                    const uint16_t *src = (const uint16_t *)(smem + 2 * buf + b * dgb + r * (kRcDgLd * 2)) + q8 * 32 + gate;
                    uint32_t w[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) w[q] = (uint32_t)src[8 * q] | ((uint32_t)src[8 * q + 4] << 16);
                    *(uint4 *)(at_row(a.dG, t, sg) + (size_t)(row0 + r) * 4 * H + gate * H + ct * 32 + q8 * 8) =
                        make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
    } else {
        if constexpr (NT > 1) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRcRegsBwd));
        load_weights();
        const int u0 = (int)ct * 32 + warp * 8, u = u0 + g;
        const bool warp_on = u0 < H;
        const int uc = warp_on ? u : 0;  // (lanes past H compute on unit 0's data and write nothing)
        // this lane's cells: unit u, rows 2 t4 + e of each N tile
        int rc[NT][2];
        bool on[NT][2];
        int s1[NT][2], s[NT][2], sn[NT][2];  // top[t + 1] (the final top first), top[t], top[t - 1]
        float v[NT][2];                      // gradient of the state s1
        float dcp[NT][2], cp[NT][2];         // dc and c of the state step t + 1 read
        float cr[NT][2], dcr[NT][2], dhs[NT][2];
        float cd[NT][2], dhd[NT][2];         // p.dead: c and gradient of the state t + 1
        uint2 gq[NT][2];
        // operands of the pointwise backward of step t, which reads row iw
        auto load_ops = [&](int t, const int (&iw)[NT][2]) {
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const size_t o = (size_t)rc[n][e] * H + uc;
                    cr[n][e] = __ldcg(at_row(a.hist_c, iw[n][e], sc) + o);
                    dcr[n][e] = __ldcg(at_row(a.dhist_c, iw[n][e], sc) + o);
                    cd[n][e] = dhd[n][e] = 0.0f;
                    if (p.dead) {
                        cd[n][e] = __ldcg(at_row(a.hist_c, t + 1, sc) + o);
                        dhd[n][e] = __ldcg(at_row(a.dhist_h, t + 1, sc) + o);
                    }
                    gq[n][e] = __ldcg((const uint2 *)(at_row(a.gates, t, sg) + o * 4));
                }
        };
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 8 * n + 2 * t4 + e;
                on[n][e] = warp_on && r < nrows;
                rc[n][e] = row0 + min(r, nrows - 1);
                s1[n][e] = p.ftop[rc[n][e]];
                s[n][e] = at_row(a.top, T - 1, si)[rc[n][e]];
                sn[n][e] = T >= 2 ? at_row(a.top, T - 2, si)[rc[n][e]] : 0;
                // the final top's gradient: what dhist_h holds already, and the loss's
                float *d = at_row(a.dhist_h, s1[n][e], sc) + (size_t)rc[n][e] * H + uc;
                float x = __ldcg(d);
                if (p.d_top) x += p.d_top[(size_t)rc[n][e] * H + uc];
                if (on[n][e]) *d = x;
                v[n][e] = x;
                dcp[n][e] = 0.0f;
                cp[n][e] = __ldcg(at_row(a.hist_c, s1[n][e], sc) + (size_t)rc[n][e] * H + uc);
                dhs[n][e] = s[n][e] == s1[n][e] ? x : __ldcg(at_row(a.dhist_h, s[n][e], sc) + (size_t)rc[n][e] * H + uc);
            }
        load_ops(T - 1, s);
        bool ok = true;
        for (int t = T - 1; t >= 0; --t) {
            const int b = t & 1;
            // Pointwise backward of step t. Its state t + 1 is the one step t + 1 read, whose c
            // and gradients are at hand; else no step read it, and its gradient is zero (or
            // what push-only mode seeded).
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 g01 = __half22float2(*(const __half2 *)&gq[n][e].x);
                    const float2 g23 = __half22float2(*(const __half2 *)&gq[n][e].y);
                    const float ig = g01.x, fg = g01.y, gg = g23.x, og = g23.y;
                    const bool live = s1[n][e] == t + 1;
                    const float dh = live ? v[n][e] : dhd[n][e], dct = live ? dcp[n][e] : 0.0f;
                    const float tcn = tanh_hw(live ? cp[n][e] : cd[n][e]);
                    const float dc = dct + dh * og * (1.0f - tcn * tcn);
                    const float di = dc * gg * ig * (1.0f - ig), df = dc * cr[n][e] * fg * (1.0f - fg);
                    const float dg = dc * ig * (1.0f - gg * gg), dq = dh * tcn * og * (1.0f - og);
                    dcp[n][e] = dcr[n][e] + dc * fg;
                    cp[n][e] = cr[n][e];
                    if (on[n][e])  // this unit's four gates of the row, K index 4 (8 warp + g) + gate
                        *(uint2 *)(smem + 2 * buf + b * dgb + (8 * n + 2 * t4 + e) * (kRcDgLd * 2) + (8 * warp + g) * 8) =
                            make_uint2(pack2_bf16(di, df), pack2_bf16(dg, dq));
                }
            // dG_t is complete; a warp whose wait ran out ends the loop for the whole CTA here
            if (__syncthreads_or(!ok)) break;
            contract(b);
            // while the parts travel: the cell gradient of the state read, the next step's operands
            float dhn[NT][2];
            int s2[NT][2];
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const size_t o = (size_t)rc[n][e] * H + uc;
                    if (on[n][e]) *(at_row(a.dhist_c, s[n][e], sc) + o) = dcp[n][e];
                    dhn[n][e] = __ldcg(at_row(a.dhist_h, sn[n][e], sc) + o);
                    s2[n][e] = at_row(a.top, max(t - 2, 0), si)[rc[n][e]];
                }
            if (t >= 1) load_ops(t - 1, sn);
            // dh_read of this CTA's units: the parts in CTA order (phase (T - 1 - t) / 2 of buffer t % 2)
            ok = rc_wait<true>(s_bar + 8 * b, (uint32_t)((T - 1 - t) >> 1) & 1, limit, abort, a.err);
            // (after a wait that ran out the phase is still open: no second arrival on it)
            if (ok && tid == 0 && t >= 2) tc::mbar_arrive_expect_tx(&rbar[b], r_bytes);
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                // M tile warp / 2, its rows g (warp even) or g + 8: the fragment's first or second pair
                const uint8_t *src = smem + b * buf + (warp >> 1) * slot + n * 512 + lane * 16 + (warp & 1) * 8;
                float2 x[8];
#pragma unroll
                for (uint32_t c = 0; c < 8; ++c) x[c] = c < C ? *(const float2 *)(src + c * 2 * slot) : make_float2(0.f, 0.f);
                float sum[2] = {x[0].x, x[0].y};
#pragma unroll
                for (uint32_t c = 1; c < 8; ++c)
                    if (c < C) {
                        sum[0] += x[c].x;
                        sum[1] += x[c].y;
                    }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    v[n][e] = dhs[n][e] + sum[e];
                    if (on[n][e]) *(at_row(a.dhist_h, s[n][e], sc) + (size_t)rc[n][e] * H + uc) = v[n][e];
                    dhs[n][e] = sn[n][e] == s[n][e] ? v[n][e] : dhn[n][e];
                    s1[n][e] = s[n][e];
                    s[n][e] = sn[n][e];
                    sn[n][e] = s2[n][e];
                }
            }
        }
    }
    rc_leave(abort);
}

// -------------------------------------------------------------------------- plan
// contraction steps of 16 the kernels are built for: the least that covers H
int rc_k(int H) { return H <= 64 ? 4 : H <= 128 ? 8 : H <= 208 ? 13 : 16; }

template <int K>
const void *rc_fn_k(bool fwd, int NT)
{
    if (fwd) return NT == 1 ? (const void *)step_rows<K, 1> : (const void *)step_rows<K, 2>;
    return NT == 1 ? (const void *)step_rowsb<K, 1> : (const void *)step_rowsb<K, 2>;
}
const void *rc_fn(bool fwd, int H, int NT)
{
    switch (rc_k(H)) {
    case 4: return rc_fn_k<4>(fwd, NT);
    case 8: return rc_fn_k<8>(fwd, NT);
    case 13: return rc_fn_k<13>(fwd, NT);
    default: return rc_fn_k<16>(fwd, NT);
    }
}

void rc_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *at, int clusters, int C, uint32_t smem, cudaStream_t st)
{
    *cfg = {};
    cfg->gridDim = dim3(clusters * C);
    cfg->blockDim = dim3(kRcThreads);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
}

// One direction with NT 8-row N tiles a cluster: every cluster co-resident (two CTAs an SM, one
// where the input is wide), or the plan is off. At H = 200 that is 38 clusters: NT = 1, 304 rows,
// 0.96 / 1.03 us a step up to 14 clusters (one CTA an SM) and 1.34 / 1.50 beyond, against 1.6 / 2.3
// of the 64-row clusters; NT = 2, 608 rows at 2.63 / 2.51, against 4.02 / 6.05 of the persistent
// kernels (the 64-row clusters reach 448 rows). A second round of clusters pays for training but
// not for a forward alone: 768 rows 4.85 / 4.68 against 4.15 / 6.12, 1024 rows 5.09 / 4.96 against
// 4.55 / 6.14. At the reach of other widths (I = H, passes of 60 steps, us, before and here): H = 32,
// 64 rows 237 / 116, 2400 (NT = 1) 505 / 186, 3500 (NT = 2) 528 / 266; H = 64, 1000 rows 522 / 189, 1400
// 531 / 252; H = 104, 448 rows 285 / 169, 900 627 / 275; H = 128, 512 rows 282 / 182, 800 585 / 281; H = 136,
// 448 rows 297 / 211, 560 646 / 342; H = 256, 288 rows 322 / 257. I = 640, H = 256: 64 rows 418 / 207.
bool rc_plan(stacklstm *s, bool fwd, int NT, PersistPlan *pl)
{
    pl->on = 0;
    // test hooks (include/stacklstm.h)
    const char *env = getenv(fwd ? "STACKLSTM_FWD_CLUSTER" : "STACKLSTM_BWD_CLUSTER");
    if (env && atoi(env) == 0) return false;
    const char *rows = getenv("STACKLSTM_ROW_CLUSTER");
    if (rows && atoi(rows) == 0) return false;
    const int C = (int)ceil_div(s->H, 32), KX = (int)ceil_div(s->I, 16);
    if (C > 8) return false;
    const int NR = 8 * NT;
    const uint32_t smem = fwd ? rc_fwd_smem(KX, rc_k(s->H), NT) : rc_bwd_smem(C, NT);
    if (smem > kSmemCap) return false;
    const void *fn = rc_fn(fwd, s->H, NT);
    cudaFuncAttributes fa;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    rc_config(&cfg, at, 1, C, smem, nullptr);
    int clusters = 0, per_sm = 0;
    // (the forward's split of the registers draws on what the block is launched with)
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess ||
        ((fwd || NT > 1) && fa.numRegs * kRcThreads < (kRcRegsStep + kRcRegsX) * (kRcThreads / 2)) ||
        smem_at_least(fn, smem) != cudaSuccess || cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kRcThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if ((int)ceil_div(s->B, NR) > clusters) return false;
    pl->on = 1;
    pl->U = 32;
    pl->EP = 1;
    pl->n_ct = pl->cl = C;
    pl->slot = (int)ceil_div(s->B, NR);
    pl->rows = NR;
    pl->smem = smem;
    pl->threads = kRcThreads;
    pl->per_sm = per_sm;  // two, or one where W_x takes over half of the shared memory
    // (clusters that could share SMs though each CTA can have one: the clear goes ahead of the steps)
    pl->spread = per_sm > 1 && s->B > NR && per_sm * (int)ceil_div(s->B, NR) <= clusters;
    return true;
}

RcArgs rc_args(stacklstm *s, const StepArgs &a, bool fwd, const float *d_top)
{
    RcArgs p{};
    p.s = a;
    p.wfrag = (const uint4 *)(fwd ? s->w_rh : s->w_rb);
    p.wx = (const uint8_t *)s->w_rx;
    p.x = (const __nv_bfloat16 *)s->x_saved;
    p.y = (__nv_bfloat16 *)s->y_direct;
    p.d_top = d_top;
    p.ftop = (s->push_only ? s->vy : s->top) + (size_t)s->T * s->B;
    p.KX = (int)ceil_div(s->I, 16);
    p.dead = s->push_only;
    return p;
}

cudaError_t rc_launch(stacklstm *const *hs, const StepArgs *as, const float *const *d_top, int n, bool fwd,
                      cudaStream_t st)
{
    RcGroup G{};
    const PersistPlan &p0 = fwd ? hs[0]->fr : hs[0]->br;
    G.n = n;
    G.C = p0.cl;
    uint32_t smem = 0;
    for (int m = 0; m < n; ++m) {
        const PersistPlan &pl = fwd ? hs[m]->fr : hs[m]->br;
        G.p[m] = rc_args(hs[m], as[m], fwd, d_top ? d_top[m] : nullptr);
        G.first[m + 1] = G.first[m] + (int)ceil_div(hs[m]->B, pl.rows);
        smem = std::max(smem, (uint32_t)pl.smem);
    }
    const void *fn = rc_fn(fwd, hs[0]->H, p0.rows / 8);
    cudaError_t e = smem_at_least(fn, smem);
    if (e) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    rc_config(&cfg, at, G.first[n], G.C, smem, st);
    void *argv[] = {(void *)&G};
    if ((e = cudaLaunchKernelExC(&cfg, fn, argv))) return e;
    hs[0]->launches += 1;
    return cudaGetLastError();
}

}  // namespace

bool bf16_plan_rows(stacklstm *s, int n_tiles)
{
    if (rc_plan(s, true, n_tiles, &s->fr) && rc_plan(s, false, n_tiles, &s->br)) return true;
    s->fr.on = s->br.on = 0;
    return false;
}

size_t bf16_rows_wh_elems(int H) { return ceil_div(H, 32) * (size_t)4 * 2 * rc_k(H) * 256; }
size_t bf16_rows_wx_elems(int I, int H) { return ceil_div(H, 32) * (size_t)128 * (ceil_div(I, 16) * 16 + 8); }
size_t bf16_rows_wb_elems(int H) { return ceil_div(H, 32) * (size_t)8 * ((rc_k(H) + 7) / 8) * 8 * 256; }
int bf16_rows_k(int H) { return rc_k(H); }

cudaError_t bf16_launch_rows(stacklstm *const *hs, const StepArgs *as, const float *const *d_top, int n, bool fwd,
                                cudaStream_t st)
{
    return rc_launch(hs, as, d_top, n, fwd, st);
}

}  // namespace sl
