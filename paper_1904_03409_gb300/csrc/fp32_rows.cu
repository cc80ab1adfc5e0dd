// fp32_rows.cu -- the fp32 path for hidden widths up to 256 (CUDA cores only, every product
// and sum in fp32): the recurrences as thread-block clusters of few rows, and the
// contractions that are not sequential as tiled ones.
//
// The gates' x part of every step, x W_x + bias, is one contraction before the steps; dx and
// dW are contractions after them. What is left in a step is h_read W_h (backward: dG W_h^T),
// whose weights a cluster of C <= 8 CTAs keeps in registers for the whole launch. Instances
// are independent, so each group of R <= 8 rows runs its T steps in a cluster of its own. A
// step is bound by what its warps issue, two a scheduler (at 64 x 200, 13 clusters of 7 CTAs
// and 5 rows: 280 two-wide multiply-adds and about 300 other instructions a warp), and by the
// exchange between the CTAs: 1.62 us forward, 1.73 backward, where a launch a step, each dot
// product reading its weights from L2 again, took 36 and 36. A 64 x 200 pass of 185 steps went
// from 20.0 ms to 1.26.
#include <stdlib.h>

#include <algorithm>

#include "common.cuh"
#include "tc.cuh"

namespace sl {
namespace {

using tc::smem_u32;

constexpr int kFrMaxW = 8, kFrThreads = 32 * kFrMaxW;  // warps of four units a CTA, at most (255 registers a thread)
constexpr long long kFrSettle = 100000;  // cycles an aborted CTA waits for stores in flight

__device__ __forceinline__ float sigmoid32(float z) { return 1.0f / (1.0f + expf(-z)); }

struct FrArgs {
    int T, B, H;
    int C, W;               // CTAs a cluster; warps of 4 units a CTA (it owns units ct 4W ..)
    const int32_t *top;     // [T + 1][B]
    float *hist_h, *hist_c; // [T + 1][B][H]
    float *gates;           // [T][B][4H]: forward, in: x W_x + bias, out: the activated gates
    float *hr;              // [T][B][H]: the state each step read (for dW)
    float *y;               // [T][B][H] step outputs, or null
    const float *wh;        // forward: W + I * 4H ([H][4H]); backward: W_h^T ([4H] rows, ldw apart)
    size_t ldw;
    float *dhist_h, *dhist_c, *dG;
    long long limit;
    int32_t *err;
};

__device__ __forceinline__ bool fr_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// bounded wait of a whole warp for bytes that the cluster's CTAs store asynchronously
__device__ __forceinline__ bool fr_wait(uint32_t bar, uint32_t parity, long long limit, volatile int *abort, int32_t *err)
{
    bool ok = fr_test(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    const long long t0 = clock64();
    while (true) {
        const bool over = clock64() - t0 >= limit || *abort;
        if (__any_sync(0xffffffffu, over)) break;
        ok = fr_test(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    *abort = 1;
    atomicCAS(err, 0, (int)SL_ERR_TIMEOUT);
    return false;
}
// no CTA leaves while another may still store into its shared memory
__device__ __forceinline__ void fr_leave(volatile int *abort)
{
    __syncthreads();
    tc::cluster_sync();
    if (*abort) {
        const long long t0 = clock64();
        while (clock64() - t0 < kFrSettle) {}
    }
    __syncthreads();
    tc::cluster_sync();
}
template <int N>
__device__ __forceinline__ void st_async_f(uint32_t addr, const float *v, uint32_t bar)
{
    static_assert(N == 1 || N == 2 || N == 4, "4, 8 or 16 bytes");
    if constexpr (N == 4)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                     "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(bar) : "memory");
    else if constexpr (N == 2)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr),
                     "f"(v[0]), "f"(v[1]), "r"(bar) : "memory");
    else
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v[0]),
                     "r"(bar) : "memory");
}
// two fused multiply-adds an instruction, each rounded as fmaf: half of what the contractions issue
__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t pair2(float lo, float hi)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ uint64_t add_2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t sub_2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ void unpair2(uint64_t v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ float add2(uint64_t v)
{
    float lo, hi;
    unpair2(v, lo, hi);
    return lo + hi;
}

// ------------------------------------------------------------------------ forward
// Warp w of CTA ct owns units u0 = 4 (ct W + w) .. + 3. Lane = (unit lane / 8, part lane % 8):
// a lane keeps its unit's four gate columns of W_h for the k of its part (float4 pieces 8 i +
// part, i < KC) and multiplies them by R rows of the h operand, 16 bytes (four k) a load: the
// warp's eight parts cover one 128-byte line of a row. The 8 parts are then summed by
// shuffles that leave each lane one row (8 / R lanes alike), whose cell it runs. The new
// operand (h' where the step pushed, else the older top) goes to every CTA of the cluster by
// st.async, a row's four units a store. Shared memory: the operand [2][R][32 KC].
template <int KC, int R>
__global__ void __launch_bounds__(kFrThreads, 1) fwd_rows_f32(FrArgs a)
{
    constexpr int KP = 32 * KC, RP = R <= 4 ? R : 8, DUP = 8 / RP;  // lanes alike per row
    __shared__ __align__(16) float s_h[2][R][KP];
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ int s_abort;
    const int T = a.T, B = a.B, H = a.H, G = 4 * H;
    const int ct = (int)tc::cluster_rank(), C = a.C, row0 = ((int)blockIdx.x / C) * R, nrows = min(R, B - row0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int u0 = 4 * (ct * a.W + warp), u = u0 + (lane >> 3), part = lane & 7;
    const bool warp_on = u0 < H, unit_on = u < H;
    const uint32_t bytes = (uint32_t)R * ((H + 3) / 4) * 16;  // of one step's operand
    volatile int *abort = &s_abort;
    for (int i = tid; i < 2 * R * KP; i += blockDim.x) (&s_h[0][0][0])[i] = 0.0f;
    if (tid == 0) {
        tc::mbar_init(&s_bar[0], 1);
        tc::mbar_init(&s_bar[1], 1);
        s_abort = 0;
        tc::fence_mbar_init();
        // the operands of steps 1 and 2 (step 0's is filled in below)
        if (T > 1) tc::mbar_arrive_expect_tx(&s_bar[1], bytes);
        if (T > 2) tc::mbar_arrive_expect_tx(&s_bar[0], bytes);
    }
    __syncthreads();
    for (int i = tid; i < nrows * H; i += blockDim.x) s_h[0][i / H][i % H] = a.hist_h[(size_t)row0 * H + i];
    uint64_t w[KC][4][2];  // [piece][gate][k pair of it]
#pragma unroll
    for (int i = 0; i < KC; ++i)
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = 4 * (8 * i + part) + q;
                v[q] = unit_on && k < H ? a.wh[(size_t)k * G + g * H + u] : 0.0f;
            }
            w[i][g][0] = pair2(v[0], v[1]);
            w[i][g][1] = pair2(v[2], v[3]);
        }
    // this lane's cell: unit u of row `row` (rows past the batch read its last row, write nothing)
    const int r = part / DUP, row = row0 + min(r, nrows - 1), uc = min(u, H - 1);
    const bool mine = unit_on && r < nrows && part % DUP == 0;
    // this lane's peers: dest and, with one lane a row, dest + 4
    const int dest = (lane >> 3) * DUP + part % DUP;
    const uint32_t self = smem_u32(&s_h[0][0][0]), bar_off = smem_u32(&s_bar[0]) - self;
    const uint32_t peer0 = tc::mapa(self, (uint32_t)min(dest, C - 1)), peer1 = tc::mapa(self, (uint32_t)min(dest + 4, C - 1));
    const bool send0 = r < R && dest < C, send1 = R > 4 && r < R && dest + 4 < C;
    const size_t cell = (size_t)row * H + uc, SB = (size_t)B * H;
    int i1 = a.top[B + row];  // top[t + 1] at step t
    float cr = a.hist_c[(size_t)a.top[row] * SB + cell], hold = a.hist_h[cell];
    float zx[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) zx[g] = a.gates[(size_t)row * G + g * H + uc];
    int i2 = a.top[(size_t)min(2, T) * B + row];
    if (mine) a.hr[cell] = hold;  // h_read(0) = h0
    __syncthreads();
    tc::cluster_sync();  // every CTA's barriers and buffers exist before any store lands on them

    for (int t = 0; t < (warp_on ? T : 0); ++t) {
        const int b = t & 1;
        __syncwarp();
        // what step t + 1 needs of rows written before this step (row t + 1 itself: unused)
        const float crn = __ldcg(a.hist_c + (size_t)i1 * SB + cell);
        const float holdn = __ldcg(a.hist_h + (size_t)i2 * SB + cell);
        const int i3 = a.top[(size_t)min(t + 3, T) * B + row];
        float zn[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) zn[g] = __ldcg(a.gates + ((size_t)min(t + 1, T - 1) * B + row) * G + g * H + uc);
        if (t > 0) {
            if (!fr_wait(smem_u32(&s_bar[b]), (uint32_t)((t - 1) >> 1) & 1, a.limit, abort, a.err)) break;
            if (tid == 0 && t + 2 < T) tc::mbar_arrive_expect_tx(&s_bar[b], bytes);
        }
        uint64_t acc2[R][4];
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
            for (int g = 0; g < 4; ++g) acc2[q][g] = 0;
#pragma unroll
        for (int i = 0; i < KC; ++i)
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const ulonglong2 h = *(const ulonglong2 *)&s_h[b][q][4 * (8 * i + part)];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    fma2(acc2[q][g], h.x, w[i][g][0]);
                    fma2(acc2[q][g], h.y, w[i][g][1]);
                }
            }
        float acc[RP][4];
#pragma unroll
        for (int q = 0; q < RP; ++q)
#pragma unroll
            for (int g = 0; g < 4; ++g) acc[q][g] = q < R ? add2(acc2[q < R ? q : 0][g]) : 0.0f;
        // sum over the parts; halving the rows kept while there are several
        float z[4];
#pragma unroll
        for (int m = 4, n = RP; m >= 1; m >>= 1, n = n > 1 ? n / 2 : 1)
#pragma unroll
            for (int q = 0; q < (n > 1 ? n / 2 : 1); ++q)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (n > 1) {
                        const float lo = acc[q][g], hi = acc[n / 2 + q][g];
                        acc[q][g] = (part & m ? hi : lo) + __shfl_xor_sync(0xffffffffu, part & m ? lo : hi, m);
                    } else {
                        acc[q][g] += __shfl_xor_sync(0xffffffffu, acc[q][g], m);
                    }
                }
#pragma unroll
        for (int g = 0; g < 4; ++g) z[g] = acc[0][g] + zx[g];
        const float ig = sigmoid32(z[0]), fg = sigmoid32(z[1]), gg = tanhf(z[2]), og = sigmoid32(z[3]);
        const float cn = fmaf(fg, cr, ig * gg), hn = og * tanhf(cn);
        const float op = !unit_on ? 0.0f : i1 == t + 1 ? hn : hold;
        if (t + 1 < T) {
            float v[4];  // the row's four units
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __shfl_sync(0xffffffffu, op, part | (j << 3));
            const uint32_t off = (uint32_t)(((b ^ 1) * R + r) * KP + u0) * 4;
            if (send0) st_async_f<4>(peer0 + off, v, peer0 + bar_off + 8 * (b ^ 1));
            if (send1) st_async_f<4>(peer1 + off, v, peer1 + bar_off + 8 * (b ^ 1));
        }
        if (mine) {
            a.hist_h[(size_t)(t + 1) * SB + cell] = hn;
            a.hist_c[(size_t)(t + 1) * SB + cell] = cn;
            if (t + 1 < T) a.hr[(size_t)(t + 1) * SB + cell] = op;
            if (a.y) a.y[(size_t)t * SB + cell] = op;
            float *gp = a.gates + ((size_t)t * B + row) * G + u;
            gp[0] = ig;
            gp[H] = fg;
            gp[2 * H] = gg;
            gp[3 * H] = og;
        }
        cr = i1 == t + 1 ? cn : crn;
        hold = i2 == t + 1 ? hn : holdn;
        i1 = i2;
        i2 = i3;
#pragma unroll
        for (int g = 0; g < 4; ++g) zx[g] = zn[g];
    }
    fr_leave(abort);
}

// ----------------------------------------------------------------------- backward
// The gate gradients of a CTA's own units stay in it: its threads multiply them by the CTA's
// 16 W gate columns of W_h (in registers: four rows of W_h by every fourth unit a thread, so
// that a 16-byte load of gate gradients feeds 16 multiply-adds) into partial dh_read values
// of all H units; thread k sends those of unit k to the CTA that owns it, which adds the
// parts in CTA order. The first 4 W R threads then hold one (unit, row) each. Shared memory: gate gradients
// [2][R][units][4 gates], parts [2][C][units][R].
template <int UP, int R>
__global__ void __launch_bounds__(kFrThreads, 1) bwd_rows_f32(FrArgs a)
{
    __shared__ __align__(16) float s_dg[2][R][UP][4];
    constexpr int RP = R <= 4 ? R : 8;  // (16-byte stores)
    __shared__ __align__(16) float s_part[2][8][UP][RP];
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ int s_abort;
    const int T = a.T, B = a.B, H = a.H, G = 4 * H, U = 4 * a.W;  // U <= UP units a CTA
    const int ct = (int)tc::cluster_rank(), C = a.C, row0 = ((int)blockIdx.x / C) * R, nrows = min(R, B - row0);
    const int tid = threadIdx.x;
    const uint32_t bytes = (uint32_t)C * max(0, min(U, H - ct * U)) * R * 4;  // of one step's parts
    volatile int *abort = &s_abort;
    for (int i = tid; i < 2 * R * UP * 4; i += blockDim.x) (&s_dg[0][0][0][0])[i] = 0.0f;
    if (tid == 0) {
        tc::mbar_init(&s_bar[0], 1);
        tc::mbar_init(&s_bar[1], 1);
        s_abort = 0;
        tc::fence_mbar_init();
        for (int i = 0; i < 2 && i < T; ++i) tc::mbar_arrive_expect_tx(&s_bar[(T - 1 - i) & 1], bytes);
    }
    const bool k_on = tid < H;
    // this thread's tile: rows 4 (tid / 4) .. + 3 of W_h by the CTA's units 4 j + tid % 4
    const int q4 = tid & 3;
    uint64_t w[UP / 4][4][2];  // [unit][row][gate pair]
#pragma unroll
    for (int j = 0; j < UP / 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float v[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int un = 4 * j + q4, k = (tid & ~3) + i;
                v[g] = k < H && un < U && ct * U + un < H ? a.wh[(size_t)(g * H + ct * U + un) * a.ldw + k] : 0.0f;
            }
            w[j][i][0] = pair2(v[0], v[1]);
            w[j][i][1] = pair2(v[2], v[3]);
        }
    const int owner = k_on ? tid / U : 0;
    const uint32_t peer = tc::mapa(smem_u32(&s_part[0][ct][k_on ? tid % U : 0][0]), (uint32_t)owner);
    const uint32_t peer_bar = tc::mapa(smem_u32(&s_bar[0]), (uint32_t)owner);
    // this thread's cell: unit ul of the CTA, row r of the group
    const int ul = tid / R, r = tid % R;
    const bool cell_on = ul < U && ct * U + ul < H, mine = cell_on && r < nrows;
    const int u = cell_on ? ct * U + ul : 0, row = row0 + min(r, nrows - 1);
    const size_t cell = (size_t)row * H + u, SB = (size_t)B * H;
    const int32_t *ltop = a.top + row;
    int s1 = ltop[(size_t)T * B], s = ltop[(size_t)(T - 1) * B], sn = ltop[(size_t)max(T - 2, 0) * B];
    float v = 0.0f, dcp = 0.0f, cp = 0.0f, cr = 0.0f, dcr = 0.0f, dhs = 0.0f, gq[4] = {};
    auto load_ops = [&](int t, int iw) {
        cr = __ldcg(a.hist_c + (size_t)iw * SB + cell);
        dcr = __ldcg(a.dhist_c + (size_t)iw * SB + cell);
#pragma unroll
        for (int g = 0; g < 4; ++g) gq[g] = __ldcg(a.gates + ((size_t)t * B + row) * G + g * H + u);
    };
    if (cell_on) {
        v = a.dhist_h[(size_t)s1 * SB + cell];  // the seeded gradient of the final top
        cp = a.hist_c[(size_t)s1 * SB + cell];
        dhs = a.dhist_h[(size_t)s * SB + cell];
        load_ops(T - 1, s);
    }
    __syncthreads();
    tc::cluster_sync();

    bool ok = true;
    for (int t = T - 1; t >= 0; --t) {
        const int b = t & 1;
        if (cell_on) {
            // pointwise backward of step t: its state t + 1 is the one step t + 1 read, or one
            // that nothing read (zero gradient)
            const float ig = gq[0], fg = gq[1], gg = gq[2], og = gq[3];
            const bool live = s1 == t + 1;
            const float dh = live ? v : 0.0f, dct = live ? dcp : 0.0f;
            const float tcn = tanhf(cp);
            const float dc = dct + dh * og * (1.0f - tcn * tcn);
            const float4 d = make_float4(dc * gg * ig * (1.0f - ig), dc * cr * fg * (1.0f - fg), dc * ig * (1.0f - gg * gg),
                                         dh * tcn * og * (1.0f - og));
            dcp = dcr + dc * fg;
            cp = cr;
            if (mine) {
                *(float4 *)s_dg[b][r][ul] = d;
                a.dhist_c[(size_t)s * SB + cell] = dcp;
                float *gp = a.dG + ((size_t)t * B + row) * G + u;
                gp[0] = d.x;
                gp[H] = d.y;
                gp[2 * H] = d.z;
                gp[3 * H] = d.w;
            }
        }
        // dG_t is complete; a warp whose wait ran out ends the loop for the whole CTA here
        if (__syncthreads_or(!ok)) break;
        // step t - 1's operands (dhist_h of the row this step adds to: taken from v below)
        float dhn = 0.0f;
        int s2 = 0;
        if (cell_on) {
            dhn = __ldcg(a.dhist_h + (size_t)sn * SB + cell);
            s2 = ltop[(size_t)max(t - 2, 0) * B];
            if (t >= 1) load_ops(t - 1, sn);
        }
        {
            uint64_t acc2[4][R];  // [row of W_h][row]
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < R; ++q) acc2[i][q] = 0;
#pragma unroll
            for (int j = 0; j < UP / 4; ++j)
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const ulonglong2 d = *(const ulonglong2 *)s_dg[b][q][4 * j + q4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        fma2(acc2[i][q], d.x, w[j][i][0]);
                        fma2(acc2[i][q], d.y, w[j][i][1]);
                    }
                }
            float acc[4][R];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < R; ++q) acc[i][q] = add2(acc2[i][q]);
            // the four threads' sums, each keeping the row of W_h that is its own (tid)
            float p2[2][R], p[R];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const float keep = q4 & 2 ? acc[2 + i][q] : acc[i][q], give = q4 & 2 ? acc[i][q] : acc[2 + i][q];
                    p2[i][q] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
                }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const float keep = q4 & 1 ? p2[1][q] : p2[0][q], give = q4 & 1 ? p2[0][q] : p2[1][q];
                p[q] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
            }
            if (k_on) {
                const uint32_t dst = peer + b * (uint32_t)sizeof(s_part[0]), bar = peer_bar + 8 * b;
                st_async_f<R >= 4 ? 4 : R>(dst, p, bar);
                if constexpr (R > 4) st_async_f<R - 4>(dst + 16, p + 4, bar);
            }
        }
        __syncwarp();
        ok = fr_wait(smem_u32(&s_bar[b]), (uint32_t)((T - 1 - t) >> 1) & 1, a.limit, abort, a.err);
        // (after a wait that ran out the phase is still open: no second arrival on it)
        if (ok && tid == 0 && t >= 2) tc::mbar_arrive_expect_tx(&s_bar[b], bytes);
        if (cell_on) {
            float x[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) x[c] = c < C ? s_part[b][c][ul][r] : 0.0f;
            float sum = x[0];
#pragma unroll
            for (int c = 1; c < 8; ++c)
                if (c < C) sum += x[c];
            v = dhs + sum;
            if (mine) a.dhist_h[(size_t)s * SB + cell] = v;
            dhs = sn == s ? v : dhn;
            s1 = s;
            s = sn;
            sn = s2;
        }
    }
    fr_leave(abort);
}

// ------------------------------------------------------------- tiled contractions
__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src, uint32_t src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

struct GemmF32 {
    int M, N, K;
    const float *A;      // [M][K] rows lda apart; kAT: its transpose, [K][M1] rows lda apart,
    const float *A2;     // and [K][M2 - M1] rows lda2 apart, the rows of A from M1; ones from M2
    int M1, M2;
    size_t lda, lda2;
    const float *B;      // [K][N] rows ldb apart, a multiple of 4, of at least N rounded up to 4
    size_t ldb;
    const float *bias;   // [N] or null
    float *C;            // [M][N] rows ldc apart; slab z of it
    float *Cr;           // kAT: the sums' rounding errors, laid out as C
    size_t ldc, slab;
};

// a float4, not four floats: it is the source of 16-byte copies
__device__ const float4 kOnes = {1.0f, 1.0f, 1.0f, 1.0f};
static_assert(alignof(decltype(kOnes)) >= 16, "kOnes is copied 16 bytes at a time");

// C = A B (+ bias) in fp32: WM x WN warps of 4 TM x 64 outputs, TM x 8 of them a thread. Blocks
// of 16 terms arrive in a ring of asynchronous copies (of EA = 4 elements where A's rows are
// aligned to that, else of one). grid z splits K evenly. Bound by the multiply-add units, which
// are busy 64% of the time (8 x 8 outputs a thread, two warps a scheduler; the pairs' duplicated
// operand costs a move each): 11840 x 800 outputs of 200 terms 90 us, 42 TFLOP/s, where 256 threads
// of 4 x 8 outputs with loads through registers reached 27; one-wide multiply-adds lose a fifth.
//
// x W_x and dx: partial sums over every 32 terms are added to a second accumulator, which keeps a
// sum of a few hundred terms near the error of its short pieces.
//
// dW and dbias (kAT) sum over all T B rows, so they are compensated, and the rounding errors go
// out beside the sums: for every two terms u = s + p + q, the error (s - u) + p + q, whose fused
// multiply-adds take the products exactly, is added to a sum of errors. That is six instructions
// for two terms instead of two. The sums alone (operands taken as they are, 1 thousand to 60
// thousand rows) then have a relative error of 3.5e-8 to 3.8e-8, that of rounding the result, as
// sums that compensated every addition had (3.5e-8 to 3.7e-8); by fours it is 4.3e-8 to 4.5e-8, and
// sums of 32 with only the splits compensated had 1.2e-7 to 1.6e-7, growing with the rows.
template <int WM, int WN, int TM, bool kAT, int EA>
__global__ void __launch_bounds__(32 * WM * WN, 8 / (WM * WN)) gemm_f32(const __grid_constant__ GemmF32 g)
{
    constexpr int NT = 32 * WM * WN, BM = WM * 4 * TM, BN = WN * 64, BK = 16, NS = TM == 8 ? 3 : 6;
    constexpr int LDA = kAT ? BM : BK + 4;                 // padded rows: four rows' 16 bytes in distinct banks
    constexpr int SA = kAT ? BK * BM : BM * LDA, SB = BK * BN;
    constexpr int NA = BM * BK / EA / NT, NB = BN * BK / 4 / NT;  // copies a thread and block
    static_assert(NA * EA * NT == BM * BK && NB * 4 * NT == BN * BK && TM % 4 == 0, "whole copies");
    __shared__ __align__(16) float sa[NS][SA], sb[NS][SB];
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, tx = lane % 8, ty = lane / 8;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN, wm = warp / WN * 4 * TM, wn = warp % WN * 64;
    const int KS = (g.K + BK - 1) / BK, z = blockIdx.z, nz = gridDim.z;
    const int k_lo = (int)((long long)KS * z / nz) * BK, k_hi = min(g.K, (int)((long long)KS * (z + 1) / nz) * BK);

    // rows and columns past the ends read the last ones' place instead and are not stored; terms
    // past k_hi are zeros
    auto load = [&](int k0, int st) {
        const bool whole = k0 + BK <= k_hi;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int c = tid + NT * i;
            const float *src;
            uint32_t dst, bytes = 4 * EA;
            if constexpr (kAT) {
                const int k = c / (BM / EA), m = c % (BM / EA) * EA, mm = m0 + m < g.M ? m0 + m : 0;
                const int kk = whole || k0 + k < k_hi ? k0 + k : k_lo;
                src = mm < g.M1 ? g.A + kk * g.lda + mm : mm < g.M2 ? g.A2 + kk * g.lda2 + (mm - g.M1) : &kOnes.x;
                dst = smem_u32(&sa[st][k * LDA + m]);
                if (!whole && k0 + k >= k_hi) bytes = 0;
            } else {
                const int m = c / (BK / EA), k = c % (BK / EA) * EA;
                src = g.A + (size_t)min(m0 + m, g.M - 1) * g.lda + k_lo;
                if (whole || k0 + k < k_hi) src += k0 + k - k_lo;
                dst = smem_u32(&sa[st][m * LDA + k]);
                if (!whole) bytes = 4 * max(0, min(EA, k_hi - k0 - k));
            }
            if constexpr (EA == 4) tc::cp_async16(dst, src, bytes);
            else cp_async4(dst, src, bytes);
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int c = tid + NT * i, k = c / (BN / 4), n = c % (BN / 4) * 4;
            const bool in = whole || k0 + k < k_hi;
            const float *src = g.B + (in ? k0 + k : k_lo) * g.ldb + (n0 + n < g.N ? n0 + n : n0);
            const uint32_t dst = smem_u32(&sb[st][k * BN + n]);
            tc::cp_async16(dst, src, in ? 16 : 0);
        }
    };

    uint64_t acc[TM][4], sum[TM][4];  // pairs of columns: the terms' sums and their sums (kAT: the sums and their errors)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = sum[i][j] = 0;
    auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sum[i][j] = add_2(sum[i][j], acc[i][j]);
                acc[i][j] = 0;
            }
    };
#pragma unroll
    for (int i = 0; i < NS - 1; ++i) {
        if (k_lo + i * BK < k_hi) load(k_lo + i * BK, i);
        tc::cp_async_commit();
    }
    int st = 0, in = NS - 1;
    bool odd = false;
    for (int k0 = k_lo; k0 < k_hi; k0 += BK) {
        tc::cp_async_wait<NS - 2>();
        __syncthreads();
        if (k0 + (NS - 1) * BK < k_hi) load(k0 + (NS - 1) * BK, in);
        tc::cp_async_commit();
        const float *pa = kAT ? &sa[st][wm + 4 * ty] : &sa[st][(wm + ty) * LDA], *pb = &sb[st][wn + 4 * tx];
        auto load_b = [&](uint64_t (&bv)[4], int k) {
            *(ulonglong2 *)bv = *(const ulonglong2 *)(pb + k * BN);
            *(ulonglong2 *)(bv + 2) = *(const ulonglong2 *)(pb + k * BN + 32);
        };
        if constexpr (kAT) {
#pragma unroll
            for (int k = 0; k < BK; k += 2) {
                float av[2][TM];
                uint64_t bv[2][4];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
#pragma unroll
                    for (int i = 0; i < TM; i += 4) *(float4 *)(av[q] + i) = *(const float4 *)(pa + (k + q) * LDA + 4 * i);
                    load_b(bv[q], k + q);
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const uint64_t a0 = pair2(av[0][i], av[0][i]), a1 = pair2(av[1][i], av[1][i]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint64_t u = acc[i][j];
                        fma2(u, a0, bv[0][j]);
                        fma2(u, a1, bv[1][j]);
                        uint64_t d = sub_2(acc[i][j], u);
                        fma2(d, a0, bv[0][j]);
                        fma2(d, a1, bv[1][j]);
                        sum[i][j] = add_2(sum[i][j], d);
                        acc[i][j] = u;
                    }
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < BK; k += 4) {
                float av[TM][4];  // row ty + 4 i
#pragma unroll
                for (int i = 0; i < TM; ++i) *(float4 *)av[i] = *(const float4 *)(pa + 4 * i * LDA + k);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint64_t bv[4];
                    load_b(bv, k + q);
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const uint64_t a2 = pair2(av[i][q], av[i][q]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) fma2(acc[i][j], a2, bv[j]);
                    }
                }
            }
            if (odd) flush();
            odd = !odd;
        }
        st = st == NS - 1 ? 0 : st + 1;
        in = in == NS - 1 ? 0 : in + 1;
    }
    tc::cp_async_wait<0>();
    if constexpr (!kAT) flush();
    auto store = [&](float *out, const uint64_t (&v)[TM][4], const float *bias) {
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
            const int n = n0 + wn + 4 * tx + 8 * j;
            float bi[4] = {};
            if (bias)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (n + q < g.N) bi[q] = bias[n + q];
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int m = m0 + wm + (kAT ? 4 * ty + 16 * (i / 4) + i % 4 : ty + 4 * i);
                if (m >= g.M) continue;
                float *o = out + (size_t)m * g.ldc + n, r[4];
                unpair2(v[i][j / 2], r[0], r[1]);
                unpair2(v[i][j / 2 + 1], r[2], r[3]);
                if (n < g.N && (g.ldc % 4 | g.N % 4) == 0)
                    *(float4 *)o = make_float4(r[0] + bi[0], r[1] + bi[1], r[2] + bi[2], r[3] + bi[3]);
                else
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (n + q < g.N) o[q] = r[q] + bi[q];
            }
        }
    };
    if constexpr (kAT) {
        store(g.C + (size_t)z * g.slab, acc, nullptr);
        store(g.Cr + (size_t)z * g.slab, sum, nullptr);
    } else {
        store(g.C + (size_t)z * g.slab, sum, g.bias);
    }
}

// sums of the nz slabs in order, and of their rounding errors in err with those of the additions
// here: the first n elements to out, the rest to out2
__global__ void slab_sum_f32(size_t n, size_t n2, int nz, const float *__restrict__ part, const float *__restrict__ err,
                             size_t slab, float *__restrict__ out, float *__restrict__ out2)
{
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n + n2; e += (size_t)gridDim.x * blockDim.x) {
        float acc = 0.0f, comp = 0.0f;
        for (int z = 0; z < nz; ++z) {
            // acc + v = t + (the error of that addition), whichever is the larger
            const float v = part[(size_t)z * slab + e], t = acc + v, w = t - acc;
            comp += (acc - (t - w)) + (v - w) + err[(size_t)z * slab + e];
            acc = t;
        }
        *(e < n ? out + e : out2 + (e - n)) = acc + comp;
    }
}

// ---------------------------------------------------------------------------- host
// rows a cluster (1, 2, 4, 5, 6, 8) x contraction pieces of 32 (forward) / units a CTA (backward)
template <int KC>
const void *fwd_fn(int R)
{
    switch (R) {
    case 1: return (const void *)fwd_rows_f32<KC, 1>;
    case 2: return (const void *)fwd_rows_f32<KC, 2>;
    case 4: return (const void *)fwd_rows_f32<KC, 4>;
    case 5: return (const void *)fwd_rows_f32<KC, 5>;
    case 6: return (const void *)fwd_rows_f32<KC, 6>;
    default: return (const void *)fwd_rows_f32<KC, 8>;
    }
}
template <int UP>
const void *bwd_fn(int R)
{
    switch (R) {
    case 1: return (const void *)bwd_rows_f32<UP, 1>;
    case 2: return (const void *)bwd_rows_f32<UP, 2>;
    case 4: return (const void *)bwd_rows_f32<UP, 4>;
    case 5: return (const void *)bwd_rows_f32<UP, 5>;
    case 6: return (const void *)bwd_rows_f32<UP, 6>;
    default: return (const void *)bwd_rows_f32<UP, 8>;
    }
}
const void *fr_fn(bool fwd, int H, int W, int R)
{
    if (!fwd)
        return W <= 2 ? bwd_fn<8>(R) : W <= 4 ? bwd_fn<16>(R) : W <= 6 ? bwd_fn<24>(R) : W == 7 ? bwd_fn<28>(R)
               : bwd_fn<32>(R);
    switch ((H + 31) / 32) {
    case 1: return fwd_fn<1>(R);
    case 2: return fwd_fn<2>(R);
    case 3: return fwd_fn<3>(R);
    case 4: return fwd_fn<4>(R);
    case 5: return fwd_fn<5>(R);
    case 6: return fwd_fn<6>(R);
    case 7: return fwd_fn<7>(R);
    default: return fwd_fn<8>(R);
    }
}

// a thread per row of W_h, and per cell
int bwd_threads(int H, int W, int R) { return std::max((int)ceil_div(H, 32) * 32, (int)ceil_div(4 * W * R, 32) * 32); }

void fr_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *at, int clusters, int C, int threads, cudaStream_t st)
{
    *cfg = {};
    cfg->gridDim = dim3(clusters * C);
    cfg->blockDim = dim3(threads);
    cfg->stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
}

// 64 x 64 tiles where they give each SM a few, else 32 x 64 ones (they are a chain of copies and
// multiply-adds along K that more of them hide: 976 x 75 outputs of 400 terms 28 -> 20 us); dW
// always the latter, whose three warps a scheduler hide the compensation's chain (64 x 200, 185 steps,
// dW with dx beside it: 507 us, 578 by 64 x 64; 300 without compensation)
template <bool kAT, int EA>
void launch_gemm(stacklstm *s, const GemmF32 &g, int splits)
{
    const unsigned nt = ceil_div(g.N, 64), big = ceil_div(g.M, 64);
    if (!kAT && (size_t)big * nt * splits >= 3 * (size_t)s->num_sms)
        gemm_f32<2, 1, kAT ? 4 : 8, kAT, EA><<<dim3(big, nt, splits), 64, 0, s->stream>>>(g);
    else
        gemm_f32<2, 1, 4, kAT, EA><<<dim3(ceil_div(g.M, 32), nt, splits), 64, 0, s->stream>>>(g);
    s->launches += 1;
}
// 16-byte copies of A where its rows allow them (A, A2 and B are the caller's 16-byte aligned tensors
// or workspace, and kOnes aligns itself)
template <bool kAT>
void launch_gemm(stacklstm *s, const GemmF32 &g, int splits)
{
    if (g.lda % 4 == 0 && (!kAT || (g.lda2 | g.M1 | g.M2) % 4 == 0))
        launch_gemm<kAT, 4>(s, g, splits);
    else
        launch_gemm<kAT, 1>(s, g, splits);
}

}  // namespace

// A forward of one step runs as fwd_step_f32 where that is shorter: the clusters read W_h into
// registers for one use, and x W_x is a launch of its own (T = 1, step / clusters: 33 + 33, 4000 rows
// 28 / 34 us; 64 + 64, 20 rows 21 / 21, 8000 rows 69 / 83; 100 + 100, 128 rows 27 / 23, 512 rows 30 /
// 32; 200 + 200, 1024 rows 108 / 109; 200 + 256, 8192 rows 848 / 910; T = 2 there 1711 / 1187). The
// clusters also hold next to nothing at H <= 3 (16 + 3, 3 steps of 4000 / 20000 rows 31 / 35 and 68 / 73
// us, 4 steps 39 / 43 and 88 / 67; 16 + 1, 8 steps of 8000 rows 97 / 96, of 40000 285 / 424).
// fwd_step_f32's operand has 48 KB of shared memory.
bool fr_step_forward(int T, int B, int I, int H)
{
    if (I + H > 12 * 1024) return false;
    if (T == 1) return H <= 64 || B >= (H <= 128 ? 512 : 4096);
    return (H <= 3 && T <= 3 && B >= 4000) || (H == 1 && B > 8192);
}

// The plan: rows a cluster R and CTAs a cluster C with the least rounds x step cycles, a step
// being the warps' multiply-adds on the fullest of the SM's four schedulers plus about 1500
// cycles of cell and exchange. (Registers allow one CTA an SM for large H: at 64 x 200, 14
// clusters of 8 CTAs are in flight at once, so 13 of five rows.)
bool fp32_plan_rows(stacklstm *s)
{
    s->fr32.on = 0;
    const int H = s->H, KC = (int)ceil_div(H, 32);
    if (H > 256) return false;
    double best = 1e30;
    for (int R : {1, 2, 4, 5, 6, 8})
        for (int want = 1; want <= 8; ++want) {
            const int W = (int)ceil_div(ceil_div(H, want), 4), C = W ? (int)ceil_div(H, 4 * W) : 0;
            if (W > kFrMaxW || C != want) continue;  // every CTA owns a unit
            int clusters = 1 << 30;
            for (int dir = 0; dir < 2; ++dir) {
                cudaLaunchConfig_t cfg;
                cudaLaunchAttribute at[1];
                int n = 0;
                fr_config(&cfg, at, 1, C, dir ? bwd_threads(H, W, R) : 32 * W, nullptr);
                if (cudaOccupancyMaxActiveClusters(&n, fr_fn(dir == 0, H, W, R), &cfg) != cudaSuccess) {
                    cudaGetLastError();
                    n = 0;
                }
                clusters = std::min(clusters, n);
            }
            if (clusters < 1) continue;
            const double rounds = ceil_div(ceil_div(s->B, R), clusters);
            const double cost = rounds * (ceil_div(W, 4) * 16.0 * KC * R + (C > 1 ? 1500.0 : 1000.0));
            if (cost < best * 0.999) {
                best = cost;
                s->fr32.on = 1;
                s->fr32.cl = C;
                s->fr32.EP = W;
                s->fr32.rows = R;
            }
        }
    if (!s->fr32.on) return false;
    s->fr32_steps = fr_step_forward(s->T, s->B, s->I, H);
    // dW and dbias: splits of the T B rows for about two rounds of 64 x 64 tiles (four an SM at
    // once), at least 128 rows each
    const size_t rows = (size_t)s->T * s->B, tiles = ceil_div(s->I + H + 1, 64) * ceil_div(4 * H, 64);
    s->fr32_split = (int)std::max<size_t>(1, std::min<size_t>(std::min<size_t>(8 * s->num_sms / tiles, rows / 128), 64));
    void *p;
    const size_t slab = ((size_t)s->I + H + 1) * 4 * H;
    const char *lim = getenv("STACKLSTM_WAIT_LIMIT_CYCLES"), *limb = getenv("STACKLSTM_WAIT_LIMIT_BWD_CYCLES");
    s->wait_limit = lim ? atoll(lim) : 4000000000LL;
    s->wait_limit_bwd = limb ? atoll(limb) : s->wait_limit;
    if (cudaMalloc(&p, 2 * sizeof(float) * slab * s->fr32_split) != cudaSuccess) {  // sums and their errors
        cudaGetLastError();
        s->fr32.on = 0;
        return false;
    }
    s->allocs.push_back(p);
    s->dw_part = (float *)p;
    return true;
}

static cudaError_t fr_launch(stacklstm *s, bool fwd, FrArgs &a)
{
    a.T = s->T; a.B = s->B; a.H = s->H;
    a.C = s->fr32.cl; a.W = s->fr32.EP;
    a.top = s->top;
    a.hist_h = (float *)s->hist_h; a.hist_c = s->hist_c;
    a.gates = (float *)s->gates; a.hr = (float *)s->a_rm; a.y = (float *)s->y_direct;
    a.dhist_h = s->dhist_h; a.dhist_c = s->dhist_c; a.dG = (float *)s->dG;
    a.limit = fwd ? s->wait_limit : s->wait_limit_bwd;
    a.err = s->err;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    fr_config(&cfg, at, (int)ceil_div(s->B, s->fr32.rows), a.C, fwd ? 32 * a.W : bwd_threads(s->H, a.W, s->fr32.rows), s->stream);
    void *argv[] = {(void *)&a};
    cudaError_t e = cudaLaunchKernelExC(&cfg, fr_fn(fwd, s->H, a.W, s->fr32.rows), argv);
    if (e) return e;
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t fp32_rows_forward(stacklstm *s, const float *x, const float *W, const float *bias)
{
    const int R = s->T * s->B, I = s->I, G = 4 * s->H;
    s->x_saved = x;
    GemmF32 g{};
    g.M = R; g.N = G; g.K = I;
    g.A = x; g.lda = I;
    g.B = W; g.ldb = G;
    g.bias = bias;
    g.C = (float *)s->gates; g.ldc = G;
    launch_gemm<false>(s, g, 1);
    FrArgs a{};
    a.wh = W + (size_t)I * G;
    return fr_launch(s, true, a);
}

cudaError_t fp32_rows_backward(stacklstm *s)
{
    FrArgs a{};
    a.wh = (const float *)s->w_fwd + s->I;  // W^T: columns I .. are W_h^T
    a.ldw = ldw_f32(s);
    return fr_launch(s, false, a);
}

cudaError_t fp32_rows_dx(stacklstm *s, float *dx)
{
    if (!dx) return cudaSuccess;
    GemmF32 g{};
    g.M = s->T * s->B; g.N = s->I; g.K = 4 * s->H;
    g.A = (const float *)s->dG; g.lda = 4 * (size_t)s->H;
    g.B = (const float *)s->w_fwd; g.ldb = ldw_f32(s);
    g.C = dx; g.ldc = s->I;
    launch_gemm<false>(s, g, 1);
    return cudaGetLastError();
}

cudaError_t fp32_rows_dw(stacklstm *s, float *dW, float *dbias)
{
    if (!dW && !dbias) return cudaSuccess;
    const int I = s->I, H = s->H, G = 4 * H, nz = s->fr32_split;
    GemmF32 g{};
    g.M1 = dW ? I : 0;
    g.M2 = dW ? I + H : 0;
    g.M = g.M2 + (dbias ? 1 : 0);  // dbias: the row of ones
    g.N = G; g.K = s->T * s->B;
    g.A = (const float *)s->x_saved; g.lda = I;
    g.A2 = (const float *)s->a_rm; g.lda2 = H;
    if (s->fr32_steps) {  // rows of [x ; h_read]
        g.A = (const float *)s->a_rm;
        g.A2 = g.A + I;
        g.lda = g.lda2 = (size_t)I + H;
    }
    g.B = (const float *)s->dG; g.ldb = G;
    g.C = s->dw_part; g.ldc = G; g.slab = (size_t)g.M * G;
    g.Cr = g.C + nz * g.slab;
    launch_gemm<true>(s, g, nz);
    slab_sum_f32<<<(unsigned)std::min<size_t>(ceil_div(g.slab, 256), (size_t)s->num_sms * 8), 256, 0, s->stream>>>(
        (size_t)g.M2 * G, g.slab - (size_t)g.M2 * G, nz, g.C, g.Cr, g.slab, dW, dbias);
    s->launches += 1;
    return cudaGetLastError();
}

}  // namespace sl
