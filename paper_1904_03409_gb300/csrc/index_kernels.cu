// index_kernels.cu -- integer bookkeeping of the homogenized step and row gathers.
//
// The prepass turns the op stream into every index the state kernels use, so the time
// loop itself never branches on an op (Algorithm 1 has no op-dependent branch):
//   p_traj[t]   pointer before step t: p_0 = 0, p_{t+1} = p_t + op_t (Sec. 3);
//   top[t]      history index of the state at slot p_t at time t: 0 is the initial state,
//               tau + 1 the state step tau wrote. Step t reads history row top[t];
//   slot_last   history index last written to each slot after the last step (-1: never).
// Every step writes slot p_t + 1 (Algorithm 1), which in history terms is row t + 1.
#include <algorithm>
#include <type_traits>
#include <map>
#include <mutex>

#include "common.cuh"

namespace sl {
namespace {

constexpr int kPrepassThreads = 32;
// shared-memory staging of prepass_walk_vec_kernel: four [32][32] int32 blocks and the ops
constexpr size_t kWalkStageBytes = 4 * 32 * 32 * 4 + 32 * 32;

// One thread per instance, walking its steps in order with the instance's stack of slot
// tags. This kernel keeps the stack in a global [T+1][B] scratch (coalesced: slot-major)
// for sequences too long for shared memory and for the allocation-free entry point;
// prepass_walk_kernel below keeps it in a column of shared memory (slot-major, so the 32
// threads of a warp hit 32 distinct banks).
__global__ void __launch_bounds__(kPrepassThreads)
prepass_kernel(int T, int B, const int8_t *__restrict__ ops, int32_t *__restrict__ p_traj,
               int32_t *__restrict__ top, int32_t *__restrict__ slot_last,
               int32_t *__restrict__ gscratch, int32_t *__restrict__ err)
{
    const int lane = threadIdx.x;
    const int b = blockIdx.x * kPrepassThreads + lane;
    if (b >= B) return;
    auto tag = [&](int slot) -> int32_t & { return gscratch[(size_t)slot * B + b]; };
    tag(0) = 0;
    for (int slot = 1; slot <= T; ++slot) tag(slot) = -1;
    int p = 0, e = SL_OK;
    // the ops of 8 steps are loaded before they are used, so that the loads do not wait on
    // one another
    int8_t opq[8];
    for (int t = 0; t < T; ++t) {
        if ((t & 7) == 0)
#pragma unroll
            for (int i = 0; i < 8; ++i) opq[i] = t + i < T ? ops[(size_t)(t + i) * B + b] : 0;
        int op = opq[t & 7];
        if (op < -1 || op > 1) {  // recorded, then run as a hold so indices stay in range
            if (e == SL_OK) e = SL_ERR_OP;
            op = 0;
        }
        if (p + op < 0) {
            if (e == SL_OK) e = SL_ERR_UNDERFLOW;
            op = 0;
        }
        p_traj[(size_t)t * B + b] = p;
        top[(size_t)t * B + b] = tag(p);
        tag(p + 1) = t + 1;  // Algorithm 1: every step writes slot p + 1
        p += op;
    }
    p_traj[(size_t)T * B + b] = p;
    top[(size_t)T * B + b] = tag(p);
    for (int slot = 0; slot <= T; ++slot) slot_last[(size_t)slot * B + b] = tag(slot);
    if (e != SL_OK) atomicCAS(err, 0, e);
}

// The push-only mode's virtual timeline (compact_kernel below), when the walk builds it.
struct VirtOut {
    int32_t *vtop, *vy, *vslot, *xidx, *vstep, *kmax;
};
// (both walks also write the caller's final pointers, p_final, when it is given)

// The same walk as prepass_kernel with the slot-tag stack in shared memory, its ops loaded
// 32 steps ahead. With kPush it also builds the push-only mode's virtual timeline in the
// same walk (what compact_kernel computes from the prepass's outputs), its real-to-virtual
// index map in shared memory beside the slot tags. (Batches of whole 32-instance blocks
// take prepass_walk_vec_kernel below.)
template <bool kPush>
__global__ void __launch_bounds__(kPrepassThreads)
prepass_walk_kernel(int T, int B, const int8_t *__restrict__ ops, int32_t *__restrict__ p_traj,
                    int32_t *__restrict__ top, int32_t *__restrict__ slot_last, int32_t *__restrict__ err, VirtOut v,
                    int32_t *__restrict__ p_final)
{
    constexpr int kBlk = 32;
    extern __shared__ int32_t s_tag[];  // [T + 1][32] slot tags, then (kPush) [T + 1][32] vmap
    const int lane = threadIdx.x;
    const int b = blockIdx.x * kPrepassThreads + lane;
    if (b >= B) return;
    int32_t *s_vmap = s_tag + (size_t)(T + 1) * kPrepassThreads;
    auto tag = [&](int slot) -> int32_t & { return s_tag[slot * kPrepassThreads + lane]; };
    // virtual index of the state at real history index j (-1: a write no step reads)
    auto vmap = [&](int j) -> int32_t & { return s_vmap[j * kPrepassThreads + lane]; };
    tag(0) = 0;
    for (int slot = 1; slot <= T; ++slot) tag(slot) = -1;
    if (kPush) {
        vmap(0) = 0;
        for (int sl = 0; sl <= T; ++sl) v.vslot[(size_t)sl * B + b] = sl == 0 ? 0 : -1;
    }
    auto load = [&](int t0, int (&q)[kBlk]) {
#pragma unroll
        for (int i = 0; i < kBlk; ++i) q[i] = t0 + i < T ? (int)ops[(size_t)(t0 + i) * B + b] : 0;
    };
    int cur[kBlk], nxt[kBlk];
    load(0, cur);
    int p = 0, e = SL_OK, k = 0;
    for (int t0 = 0; t0 < T; t0 += kBlk) {
        if (t0 + kBlk < T) load(t0 + kBlk, nxt);
#pragma unroll
        for (int i = 0; i < kBlk; ++i) {
            const int t = t0 + i;
            if (t >= T) break;
            int op = cur[i];
            if (op < -1 || op > 1) {  // recorded, then run as a hold so indices stay in range
                if (e == SL_OK) e = SL_ERR_OP;
                op = 0;
            }
            if (p + op < 0) {
                if (e == SL_OK) e = SL_ERR_UNDERFLOW;
                op = 0;
            }
            const size_t ti = (size_t)t * B + b;
            const int tp = tag(p);
            p_traj[ti] = p;
            top[ti] = tp;
            tag(p + 1) = t + 1;  // Algorithm 1: every step writes slot p + 1
            if (kPush) {
                // a state that is read is a push write or the initial state (clamp never applies)
                const int rd = max(0, vmap(tp));
                v.vy[ti] = rd;
                if (op == 1) {
                    v.xidx[(size_t)k * B + b] = t;
                    v.vtop[(size_t)k * B + b] = rd;
                    v.vstep[ti] = k;
                    vmap(t + 1) = k + 1;
                    v.vslot[(size_t)(p + 1) * B + b] = k + 1;
                    ++k;
                } else {
                    v.vstep[ti] = -1;
                    vmap(t + 1) = -1;
                }
            }
            p += op;
        }
#pragma unroll
        for (int i = 0; i < kBlk; ++i) cur[i] = nxt[i];
    }
    const int tp = tag(p);
    p_traj[(size_t)T * B + b] = p;
    top[(size_t)T * B + b] = tp;
    if (p_final) p_final[b] = p;
    for (int slot = 0; slot <= T; ++slot) slot_last[(size_t)slot * B + b] = tag(slot);
    if (kPush) {
        v.vy[(size_t)T * B + b] = max(0, vmap(tp));
        for (int kk = k; kk < T; ++kk) {
            v.xidx[(size_t)kk * B + b] = -1;
            v.vtop[(size_t)kk * B + b] = 0;
        }
        v.vtop[(size_t)T * B + b] = 0;
        atomicMax(v.kmax, k);
    }
    if (e != SL_OK) atomicCAS(err, 0, e);
}

// prepass_walk_kernel for batches of whole 32-instance blocks (B % 32 == 0, ops 4-byte
// aligned), its global traffic in 16-byte pieces: the walk costs about as much per memory
// instruction of the block's one warp as per step, so the warp loads a block of 32 steps'
// ops as 4-byte words (eight lanes a row) into shared memory, walks it there, stages the
// block's pointers and tops (and virtual indices) in shared memory, and writes them four
// rows per instruction; the slot tags go out the same way, and the push-only tables that
// are mostly -1 / 0 are written so before the walk (__syncwarp orders those stores before
// the walk's own stores to the same rows).
template <bool kPush>
__global__ void __launch_bounds__(kPrepassThreads)
prepass_walk_vec_kernel(int T, int B, const int8_t *__restrict__ ops, int32_t *__restrict__ p_traj,
                        int32_t *__restrict__ top, int32_t *__restrict__ slot_last, int32_t *__restrict__ err,
                        VirtOut v, int32_t *__restrict__ p_final)
{
    constexpr int kBlk = 32;
    // [T + 1][32] slot tags, (kPush) [T + 1][32] vmap, then the block staging:
    // pointer, top, (kPush) vy, vstep, each [32 steps][32], and the ops [32 steps][32 bytes]
    extern __shared__ int32_t s_tag[];
    const int lane = threadIdx.x, b0 = blockIdx.x * kPrepassThreads, b = b0 + lane;
    const int rq = lane >> 3, pc = 4 * (lane & 7);  // row of four, 16-byte piece: the vector pattern
    int32_t *s_vmap = s_tag + (size_t)(T + 1) * kPrepassThreads;
    int32_t *st_p = s_tag + (size_t)(kPush ? 2 : 1) * (T + 1) * kPrepassThreads;
    int32_t *st_t = st_p + kBlk * 32, *st_y = st_t + kBlk * 32, *st_v = st_y + kBlk * 32;
    uint32_t *st_o = (uint32_t *)(st_v + kBlk * 32);  // [32 steps][8 words]
    auto tag = [&](int slot) -> int32_t & { return s_tag[slot * kPrepassThreads + lane]; };
    auto vmap = [&](int j) -> int32_t & { return s_vmap[j * kPrepassThreads + lane]; };
    // rows [r0, r1) of a [rows][B] int32 table: this block's 32 columns, four rows at a time
    auto fill = [&](int32_t *dst, int r0, int r1, int val) {
        const uint4 w = make_uint4(val, val, val, val);
        for (int r = r0 + rq; r < r1; r += 4) *(uint4 *)(dst + (size_t)r * B + b0 + pc) = w;
    };
    auto flush = [&](int32_t *dst, const int32_t *src, int r0, int nrows) {  // src: [nrows][32]
        for (int r = rq; r < nrows; r += 4) *(uint4 *)(dst + (size_t)(r0 + r) * B + b0 + pc) = *(const uint4 *)(src + r * 32 + pc);
    };
    auto load = [&](int t0, uint32_t (&q)[8]) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int t = t0 + rq + 4 * j;
            q[j] = t < T ? *(const uint32_t *)(ops + (size_t)t * B + b0 + pc) : 0u;
        }
    };
    tag(0) = 0;
    for (int slot = 1; slot <= T; ++slot) tag(slot) = -1;
    if (kPush) {
        vmap(0) = 0;
        fill(v.vslot, 0, 1, 0);
        fill(v.vslot, 1, T + 1, -1);
        fill(v.xidx, 0, T, -1);
        fill(v.vtop, 0, T + 1, 0);
        __syncwarp();
    }
    uint32_t cur[8], nxt[8];
    load(0, cur);
    int p = 0, e = SL_OK, k = 0;
    for (int t0 = 0; t0 < T; t0 += kBlk) {
        if (t0 + kBlk < T) load(t0 + kBlk, nxt);
#pragma unroll
        for (int j = 0; j < 8; ++j) st_o[(rq + 4 * j) * 8 + (lane & 7)] = cur[j];
        __syncwarp();
        const int n = min(kBlk, T - t0);
        const int8_t *ob = (const int8_t *)st_o;
        for (int i = 0; i < n; ++i) {
            const int t = t0 + i;
            int op = ob[i * 32 + lane];
            if (op < -1 || op > 1) {  // recorded, then run as a hold so indices stay in range
                if (e == SL_OK) e = SL_ERR_OP;
                op = 0;
            }
            if (p + op < 0) {
                if (e == SL_OK) e = SL_ERR_UNDERFLOW;
                op = 0;
            }
            const int tp = tag(p);
            st_p[i * 32 + lane] = p;
            st_t[i * 32 + lane] = tp;
            tag(p + 1) = t + 1;  // Algorithm 1: every step writes slot p + 1
            if (kPush) {
                // a state that is read is a push write or the initial state (clamp never applies)
                const int rd = max(0, vmap(tp));
                st_y[i * 32 + lane] = rd;
                st_v[i * 32 + lane] = op == 1 ? k : -1;
                vmap(t + 1) = op == 1 ? k + 1 : -1;
                if (op == 1) {
                    v.xidx[(size_t)k * B + b] = t;
                    v.vtop[(size_t)k * B + b] = rd;
                    v.vslot[(size_t)(p + 1) * B + b] = k + 1;
                    ++k;
                }
            }
            p += op;
        }
        __syncwarp();
        flush(p_traj, st_p, t0, n);
        flush(top, st_t, t0, n);
        if (kPush) {
            flush(v.vy, st_y, t0, n);
            flush(v.vstep, st_v, t0, n);
        }
        __syncwarp();  // the staging is read before the next block overwrites it
#pragma unroll
        for (int j = 0; j < 8; ++j) cur[j] = nxt[j];
    }
    const int tp = tag(p);
    p_traj[(size_t)T * B + b] = p;
    top[(size_t)T * B + b] = tp;
    if (p_final) p_final[b] = p;
    if (kPush) {
        v.vy[(size_t)T * B + b] = max(0, vmap(tp));
        atomicMax(v.kmax, k);
    }
    __syncwarp();
    flush(slot_last, s_tag, 0, T + 1);
    if (e != SL_OK) atomicCAS(err, 0, e);
}

// out[r] = hist row (idx[r], r % B), or zeros where idx[r] < 0; rows of `pieces` values of the
// raw type E (16 bytes where the row length and the addresses allow, else 4 or 2). 2^lg lanes
// take a row, a warp (kWarp) or the fewest that give each piece one, four rows at a time, so that
// the index loads and the row loads are in flight together: bound by the bytes moved (195 x 1024
// rows of 400 bytes, 160 MB: 23 us, 115 as one thread per 2-byte value with a 64-bit division each;
// 256 x 256 rows of 2 KB: 28 us, 188; 40 x 20000 rows of 16 bytes: 10 us, 27, and 55 with a warp to
// every row).
template <typename E, bool kWarp>
__global__ void __launch_bounds__(256) gather_rows_kernel(const int32_t *__restrict__ idx, int B, int rows, int pieces,
                                                          int lg_, const E *__restrict__ hist, E *__restrict__ out)
{
    constexpr int N = 4;
    const int lg = kWarp ? 5 : lg_;
    const int lane = threadIdx.x & 31, sub = lane & ((1 << lg) - 1), per = 32 >> lg, warps = gridDim.x * (blockDim.x >> 5);
    auto source = [&](uint32_t row) -> long long {  // of one row (past the last: of that one), or -1
        const int r = (int)min(row, (uint32_t)rows - 1), s = idx[r];
        return s >= 0 ? (long long)s * B + r % B : -1;
    };
    for (int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); (long long)g * N * per < rows; g += warps) {
        const uint32_t r0 = (uint32_t)(g * N * per + (lane >> lg));
        const long long mine = kWarp ? source(r0 + (lane & (N - 1))) : 0;  // a row to each of four lanes
        const E *from[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const long long q = kWarp ? __shfl_sync(0xffffffffu, mine, i) : source(r0 + i * per);
            from[i] = q >= 0 ? hist + (size_t)q * pieces : nullptr;
        }
        for (int k = sub; k < pieces; k += 1 << lg) {
            E v[N];
#pragma unroll
            for (int i = 0; i < N; ++i) v[i] = from[i] ? from[i][k] : E{};
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (r0 + i * per < (uint32_t)rows) out[(size_t)(r0 + i * per) * pieces + k] = v[i];
        }
    }
}

// Seed the gradient history with the loss terms before the reverse loop:
// d_top_h goes to the final top, dy_t to the top after step t (Algorithm 1's output).
// One thread per (b, j); its additions run in a fixed order (final top, then t = T-1..0).
__global__ void seed_grads_kernel(int T, int B, int H, const int32_t *__restrict__ top,
                                  const float *__restrict__ d_top_h, const float *__restrict__ dy,
                                  float *__restrict__ dhist_h)
{
    const size_t n = (size_t)B * H;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
         e += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(e / H), j = (int)(e - (size_t)b * H);
        if (d_top_h) {
            const int s = top[(size_t)T * B + b];
            dhist_h[((size_t)s * B + b) * H + j] += d_top_h[e];
        }
        if (dy)
            for (int t = T - 1; t >= 0; --t) {
                const int s = top[(size_t)(t + 1) * B + b];
                dhist_h[((size_t)s * B + b) * H + j] += dy[(size_t)t * n + e];
            }
    }
}

// The same seeding with per-step gradients dy, for one instance and 32 N units per block
// (one warp, N units a lane): the sums of the T + 1 rows accumulate in shared memory in the same
// order as above (final top, then t = T-1..0), then every row is written once. The gradient
// history is zero before the seeding, so writing the sums equals adding them. A step is one
// addition to a row in shared memory (the top's row held in registers, stored and loaded at a
// change of row, took a branch a step: 256 x 1024, 256 steps, 185 us, 170 so); the loads run 24
// to 32 steps ahead, by asynchronous copies into a ring of which each lane reads back only its own
// (eight steps ahead in registers left it waiting for memory: 281 us; rings of 16 and 64 steps
// 192, 199; a block to an instance and 64 units with its rows in parallel 279).
constexpr int kSeedRing = 32, kSeedGroup = 8;  // steps in flight, steps a copy group
template <int N>
__global__ void __launch_bounds__(32) seed_grads_dy_kernel(int T, int B, int H, const int32_t *__restrict__ top,
                                                            const float *__restrict__ d_top_h,
                                                            const float *__restrict__ dy, float *__restrict__ dhist_h)
{
    struct alignas(4 * N) Vec {
        float f[N];
    };
    extern __shared__ __align__(16) uint8_t seed_smem[];
    const int lane = threadIdx.x;
    Vec *ring = (Vec *)seed_smem + lane;   // step i: ring[32 (i mod kSeedRing)]
    Vec *slot = ring + 32 * kSeedRing;     // row s: slot[32 s]
    const int b = blockIdx.x, j = (blockIdx.y * 32 + lane) * N;
    const bool on = j < H;  // (H % N == 0: whole pieces)
    const size_t step = (size_t)B * H, e = (size_t)b * H + (on ? j : 0);
    auto fetch = [&](int i0) {  // steps T - 1 - i0 ..: one copy group
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + 32 * (i0 % kSeedRing));
#pragma unroll
        for (int i = 0; i < kSeedGroup; ++i)
            if (i0 + i < T)
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst + i * 128 * N),
                             "l"(dy + (size_t)(T - 1 - i0 - i) * step + e), "n"(4 * N)
                             : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // lane l keeps the top after step T - 1 - (i0 + l), i0 a multiple of 32
    auto tops = [&](int i0) { return top[(size_t)max(T - i0 - lane, 1) * B + b]; };
    for (int i = 0; i < kSeedRing - kSeedGroup; i += kSeedGroup) fetch(i);
    int s_cur = tops(0), s_nxt = T > 32 ? tops(32) : 0;
    for (int i = lane; i < (T + 1) * 8 * N; i += 32) ((uint4 *)(slot - lane))[i] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    if (d_top_h) {
        Vec acc{};
        const Vec d = *(const Vec *)(d_top_h + e);
#pragma unroll
        for (int i = 0; i < N; ++i) acc.f[i] += d.f[i];
        slot[32 * top[(size_t)T * B + b]] = acc;
    }
    auto add = [&](int r, const Vec &g) {
        Vec acc = slot[32 * r];
#pragma unroll
        for (int k = 0; k < N; ++k) acc.f[k] += g.f[k];
        slot[32 * r] = acc;
    };
    for (int i0 = 0; i0 < T; i0 += kSeedGroup) {
        fetch(i0 + kSeedRing - kSeedGroup);
        asm volatile("cp.async.wait_group %0;" ::"n"(kSeedRing / kSeedGroup - 1) : "memory");
        // the group's gradients and rows first: only the additions stay on the chain
        int s[kSeedGroup];
        Vec g[kSeedGroup];
#pragma unroll
        for (int i = 0; i < kSeedGroup; ++i) {
            s[i] = __shfl_sync(0xffffffffu, s_cur, (i0 + i) & 31);
            g[i] = ring[32 * ((i0 + i) % kSeedRing)];
        }
        if (i0 + kSeedGroup <= T) {
#pragma unroll
            for (int i = 0; i < kSeedGroup; ++i) add(s[i], g[i]);
        } else {
#pragma unroll
            for (int i = 0; i < kSeedGroup; ++i)
                if (i0 + i < T) add(s[i], g[i]);
        }
        if ((i0 + kSeedGroup) % 32 == 0) {
            s_cur = s_nxt;
            if (i0 + kSeedGroup + 32 < T) s_nxt = tops(i0 + kSeedGroup + 32);
        }
    }
    if (on)
#pragma unroll 8
        for (int r = 0; r <= T; ++r) *(Vec *)(dhist_h + (size_t)r * step + e) = slot[32 * r];
}

// Push-only mode: the virtual timeline of each instance. By Observation 2 of Sec. 3 only
// a push step's write is ever read (a pop or hold writes slot p + 1 above the new top,
// and the next push overwrites it before the pointer gets there), so instance b's
// computation is the chain of its push steps alone: virtual step k is its k-th push, it
// reads the virtual state of the push that wrote the slot it reads (or the initial state,
// virtual index 0) and writes virtual history row k + 1. One thread per instance walks its
// steps in order, so every index it looks up was set at an earlier step. Virtual steps
// past an instance's last push read the initial state and their writes are never read.
// A step is a push when its pointer moves up by one (ops the prepass rejected ran as
// holds). vslot is the stack of Sec. 2's definition: each slot's last pushed state.
// kmax (zero on entry) receives the most pushes of any instance.
template <bool kOnChip>
__global__ void __launch_bounds__(kPrepassThreads)
compact_kernel(int T, int B, const int32_t *__restrict__ p_traj, const int32_t *__restrict__ top,
               int32_t *__restrict__ vtop, int32_t *__restrict__ gvmap,
               int32_t *__restrict__ vy, int32_t *__restrict__ vslot, int32_t *__restrict__ xidx,
               int32_t *__restrict__ vstep, int32_t *__restrict__ kmax)
{
    extern __shared__ int32_t s_vmap[];
    const int lane = threadIdx.x, b = blockIdx.x * kPrepassThreads + lane;
    if (b >= B) return;
    // vmap: the virtual index of the state at real history index j (written at step j - 1,
    // or the initial state at j = 0), -1 for a non-push write; in shared memory when it fits
    auto vmap = [&](int j) -> int32_t & {
        return kOnChip ? s_vmap[j * kPrepassThreads + lane] : gvmap[(size_t)j * B + b];
    };
    // a state that is read is always a push write or the initial state, so the clamp never
    // applies to valid prepass output
    auto vof = [&](int j) { return max(0, vmap(j)); };
    vmap(0) = 0;
    vslot[b] = 0;  // slot 0: the initial state
    for (int sl = 1; sl <= T; ++sl) vslot[(size_t)sl * B + b] = -1;
    int k = 0;
    // the tops and pointers of 8 steps are loaded before they are used
    int tq[8], pq[9];
    for (int t = 0; t < T; ++t) {
        if ((t & 7) == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                tq[i] = t + i < T ? top[(size_t)(t + i) * B + b] : 0;
                pq[i] = t + i <= T ? p_traj[(size_t)(t + i) * B + b] : 0;
            }
            pq[8] = t + 8 <= T ? p_traj[(size_t)(t + 8) * B + b] : 0;
        }
        const size_t i = (size_t)t * B + b;
        const int rd = vof(tq[t & 7]);
        vy[i] = rd;
        if (pq[(t & 7) + 1] - pq[t & 7] == 1) {
            xidx[(size_t)k * B + b] = t;
            vtop[(size_t)k * B + b] = rd;
            vstep[i] = k;
            vmap(t + 1) = k + 1;
            vslot[(size_t)(pq[t & 7] + 1) * B + b] = k + 1;
            ++k;
        } else {
            vstep[i] = -1;
            vmap(t + 1) = -1;
        }
    }
    vy[(size_t)T * B + b] = vof(top[(size_t)T * B + b]);
    for (int kk = k; kk < T; ++kk) {
        xidx[(size_t)kk * B + b] = -1;
        vtop[(size_t)kk * B + b] = 0;
    }
    vtop[(size_t)T * B + b] = 0;
    atomicMax(kmax, k);
}

// The initial state's gradients: history row 0 (slot 0 always holds the initial state). One
// launch for both; two copies are bound by their starts, 2 x 3.5 us.
__global__ void h0_grads_kernel(size_t n, const float *__restrict__ dh, const float *__restrict__ dc,
                                float *__restrict__ dh0, float *__restrict__ dc0)
{
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        if (dh0) dh0[e] = dh[e];
        if (dc0) dc0[e] = dc[e];
    }
}

// Push-only mode: dx rows of the steps that do not push are zero (a state no step reads
// has zero gradient); the push rows are written by the input-gradient contraction.
// A warp per row: the row's step index is read once, its 16-byte pieces written by the
// warp's lanes side by side.
__global__ void zero_nonpush_rows_kernel(size_t rows, int I4, const int32_t *__restrict__ vstep,
                                         float4 *__restrict__ dx)
{
    const int lane = threadIdx.x & 31;
    const size_t warps = (size_t)gridDim.x * (blockDim.x >> 5);
    for (size_t r = (size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
        if (vstep[r] >= 0) continue;
        float4 *row = dx + r * I4;
        for (int i = lane; i < I4; i += 32) row[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

}  // namespace

cudaError_t launch_compact(stacklstm *s)
{
    if (s->walk_built_virtual) return cudaSuccess;  // the prepass's walk built the timeline
    cudaError_t e = cudaMemsetAsync(s->kmax, 0, sizeof(int32_t), s->stream);
    if (e) return e;
    // the index table on chip when the prepass's slot-tag stack is (the same size)
    const unsigned grid = ceil_div(s->B, kPrepassThreads);
    if (s->prepass_smem > 0) {
        if (s->prepass_smem > 48 * 1024 &&
            (e = smem_at_least((const void *)compact_kernel<true>, (size_t)s->prepass_smem)))
            return e;
        compact_kernel<true><<<grid, kPrepassThreads, s->prepass_smem, s->stream>>>(
            s->T, s->B, s->p_traj, s->top, s->vtop, s->vmap, s->vy, s->vslot, s->xidx, s->vstep, s->kmax);
    } else {
        compact_kernel<false><<<grid, kPrepassThreads, 0, s->stream>>>(
            s->T, s->B, s->p_traj, s->top, s->vtop, s->vmap, s->vy, s->vslot, s->xidx, s->vstep, s->kmax);
    }
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t read_virtual_steps(stacklstm *s)
{
    cudaError_t e = cudaMemcpyAsync(s->kmax_host, s->kmax, sizeof(int32_t), cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e) return e;
    // at least one step, so that every kernel has work of its usual shape (a batch with no
    // push at all runs one virtual step whose write nobody reads)
    s->Tr = std::max(1, std::min(s->T, (int)*s->kmax_host));
    return cudaSuccess;
}

cudaError_t launch_h0_grads(stacklstm *s, float *dh0, float *dc0, cudaStream_t st)
{
    if (!dh0 && !dc0) return cudaSuccess;
    const size_t n = (size_t)s->B * s->H;
    h0_grads_kernel<<<std::min<unsigned>(ceil_div(n, 256), s->num_sms), 256, 0, st>>>(n, s->dhist_h, s->dhist_c, dh0, dc0);
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_zero_nonpush_rows(stacklstm *s, float *dx)
{
    if (!dx) return cudaSuccess;
    const size_t rows = (size_t)s->T * s->B;
    const int I4 = s->I / 4;  // the bf16 path has I % 8 == 0
    const unsigned grid = (unsigned)std::max<size_t>(1, std::min<size_t>(ceil_div(rows, 8), (size_t)s->num_sms * 16));
    zero_nonpush_rows_kernel<<<grid, 256, 0, s->stream>>>(rows, I4, s->vstep, (float4 *)dx);
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t smem_at_least(const void *fn, size_t bytes)
{
    static std::mutex m;
    static std::map<std::pair<int, const void *>, size_t> set;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    std::lock_guard<std::mutex> lk(m);
    size_t &cur = set[{dev, fn}];
    if (bytes <= cur) return cudaSuccess;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes))) return e;
    cur = bytes;
    return cudaSuccess;
}

// The slot-tag stack goes on chip when (T + 1) slots x 32 instances fit in shared memory.
cudaError_t configure_prepass(stacklstm *s)
{
    const size_t bytes = (size_t)(s->T + 1) * kPrepassThreads * sizeof(int32_t);
    int optin = 0;
    cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->device);
    if (e) return e;
    s->prepass_smem = 0;
    s->walk_push_smem = 0;
    if (bytes + kWalkStageBytes + 1024 <= (size_t)optin) {
        if ((e = smem_at_least((const void *)prepass_walk_kernel<false>, bytes)) ||
            (e = smem_at_least((const void *)prepass_walk_vec_kernel<false>, bytes + kWalkStageBytes)))
            return e;
        s->prepass_smem = (int)bytes;
        // the push-only walk keeps the real-to-virtual index map beside the slot tags
        if (2 * bytes + kWalkStageBytes + 1024 <= (size_t)optin) {
            if ((e = smem_at_least((const void *)prepass_walk_kernel<true>, 2 * bytes)) ||
                (e = smem_at_least((const void *)prepass_walk_vec_kernel<true>, 2 * bytes + kWalkStageBytes)))
                return e;
            s->walk_push_smem = (int)(2 * bytes);
        }
    }
    return cudaSuccess;
}

cudaError_t launch_prepass(stacklstm *s, const int8_t *ops, int32_t *p_final)
{
    const unsigned grid = ceil_div(s->B, kPrepassThreads);
    s->walk_built_virtual = 0;
    s->pfinal_written = s->prepass_smem > 0;  // the walks write it; prepass_kernel does not
    // whole 32-instance blocks and word-aligned ops: the walk's traffic in 16-byte pieces
    const bool vec = s->B % kPrepassThreads == 0 && ((uintptr_t)ops & 3) == 0;
    if (s->push_only && s->walk_push_smem > 0) {
        cudaError_t e = cudaMemsetAsync(s->kmax, 0, sizeof(int32_t), s->stream);
        if (e) return e;
        const VirtOut v{s->vtop, s->vy, s->vslot, s->xidx, s->vstep, s->kmax};
        if (vec)
            prepass_walk_vec_kernel<true><<<grid, kPrepassThreads, s->walk_push_smem + kWalkStageBytes, s->stream>>>(
                s->T, s->B, ops, s->p_traj, s->top, s->slot_last, s->err, v, p_final);
        else
            prepass_walk_kernel<true><<<grid, kPrepassThreads, s->walk_push_smem, s->stream>>>(
                s->T, s->B, ops, s->p_traj, s->top, s->slot_last, s->err, v, p_final);
        s->walk_built_virtual = 1;
    } else if (s->prepass_smem > 0) {
        if (vec)
            prepass_walk_vec_kernel<false><<<grid, kPrepassThreads, s->prepass_smem + kWalkStageBytes, s->stream>>>(
                s->T, s->B, ops, s->p_traj, s->top, s->slot_last, s->err, VirtOut{}, p_final);
        else
            prepass_walk_kernel<false><<<grid, kPrepassThreads, s->prepass_smem, s->stream>>>(
                s->T, s->B, ops, s->p_traj, s->top, s->slot_last, s->err, VirtOut{}, p_final);
    } else {
        prepass_kernel<<<grid, kPrepassThreads, 0, s->stream>>>(s->T, s->B, ops, s->p_traj, s->top, s->slot_last,
                                                                s->slot_scratch, s->err);
    }
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_gather_rows(stacklstm *s, const int32_t *idx, int rows, size_t elem_bytes,
                               const void *hist, void *out, int row_elems)
{
    if (rows == 0 || row_elems == 0) return cudaSuccess;
    // (hist is workspace and out 16-byte aligned: a row whose length is a multiple of 16 bytes is too)
    const size_t row_bytes = (size_t)row_elems * elem_bytes;
    const int pieces = row_bytes % 16 == 0 ? (int)(row_bytes / 16) : row_elems;
    int lg = 0;
    while (lg < 5 && 1 << lg < pieces) ++lg;
    const unsigned grid = (unsigned)std::min<size_t>(ceil_div(rows, 1024 >> lg), (size_t)s->num_sms * 16);
    auto go = [&](auto *of) {
        using E = std::remove_pointer_t<decltype(of)>;
        if (lg == 5)
            gather_rows_kernel<E, true><<<grid, 256, 0, s->stream>>>(idx, s->B, rows, pieces, lg, (const E *)hist, (E *)out);
        else
            gather_rows_kernel<E, false><<<grid, 256, 0, s->stream>>>(idx, s->B, rows, pieces, lg, (const E *)hist, (E *)out);
    };
    if (row_bytes % 16 == 0)
        go((uint4 *)nullptr);
    else if (elem_bytes == 4)
        go((uint32_t *)nullptr);
    else
        go((uint16_t *)nullptr);
    s->launches += 1;
    return cudaGetLastError();
}

template <int N>
static cudaError_t seed_dy(stacklstm *s, size_t bytes, const int32_t *top, const float *d_top_h, const float *dy)
{
    const cudaError_t e = smem_at_least((const void *)seed_grads_dy_kernel<N>, bytes);
    if (e) return e;
    seed_grads_dy_kernel<N><<<dim3(s->B, ceil_div(s->H, 32 * N)), 32, bytes, s->stream>>>(s->T, s->B, s->H, top, d_top_h,
                                                                                          dy, s->dhist_h);
    s->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_seed_grads(stacklstm *s, const float *d_top_h, const float *dy)
{
    if (!d_top_h && !dy) return cudaSuccess;
    const int32_t *top = s->push_only ? s->vy : s->top;
    // Units a lane: four while four warps' rows fit on an SM, two while three do, if that divides H
    // and the blocks then cover no more units past H. (us with 1 / 2 / 4: 512 x 256, 60 steps 26 / 23 /
    // 22, 120 steps 43 / 39 / 48; 256 x 1024, 256 steps 184 / 177 / 281; 64 x 256, 300 steps 24 / 25 / 28;
    // 1024 x 200, 195 steps, where two and four cover 256 units 151 / 159 / 230; 2000 x 32, 40 steps 13 /
    // 19 / 25)
    const size_t acc_bytes = (size_t)(s->T + 1 + kSeedRing) * 32 * sizeof(float);
    auto fits = [&](int N, size_t cap) {
        return s->H % N == 0 && N * acc_bytes <= cap && ceil_div(s->H, 32 * N) * N <= ceil_div(s->H, 32);
    };
    // (200 KB of rows and the ring, 4 KB: sequences of up to 1599 steps)
    if (dy && acc_bytes <= 204 * 1024) {
        if (fits(4, 56 * 1024)) return seed_dy<4>(s, 4 * acc_bytes, top, d_top_h, dy);
        if (fits(2, 75 * 1024)) return seed_dy<2>(s, 2 * acc_bytes, top, d_top_h, dy);
        return seed_dy<1>(s, acc_bytes, top, d_top_h, dy);
    }
    const size_t n = (size_t)s->B * s->H;
    const unsigned grid = (unsigned)std::min<size_t>(ceil_div(n, 256), (size_t)s->num_sms * 16);
    // the (virtual, in push-only mode) history index of the top at each real time
    seed_grads_kernel<<<grid, 256, 0, s->stream>>>(s->T, s->B, s->H, top, d_top_h, dy, s->dhist_h);
    s->launches += 1;
    return cudaGetLastError();
}

// ------------------------------------------------------------ allocation-free prepass
// stacklstm_pointers_noalloc runs the prepass above for callers that cannot allocate
// device memory. Its scratch (the slot-tag stack, the last-writer table and a status
// word) is this file-scope array, which every GPU that loads the library holds until
// the process exits. Every call shares it and it keeps the last call's contents.
namespace {
constexpr size_t kNoAllocMaxSlots = (size_t)1 << 20;  // (T + 1) * B at most
constexpr int kNoAllocMaxDevices = 64;
__device__ __align__(256) int32_t g_noalloc_scratch[2 * kNoAllocMaxSlots + 64];

std::mutex g_noalloc_mu;
int32_t *g_noalloc_addr[kNoAllocMaxDevices] = {};

// Device address of the scratch on the current device (the host-side name of the array
// is only a stand-in). Looked up once per device.
cudaError_t noalloc_scratch(int32_t **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        if ((e = cudaGetSymbolAddress(&p, g_noalloc_scratch)) != cudaSuccess) return e;
        g_noalloc_addr[dev] = (int32_t *)p;
    }
    *out = g_noalloc_addr[dev];
    return cudaSuccess;
}
}  // namespace
}  // namespace sl

extern "C" sl_status stacklstm_pointers_noalloc(int T, int B, const int8_t *ops, int32_t *p_traj, int32_t *src,
                                                void *stream)
{
    using namespace sl;
    if (T < 1 || B < 1 || !ops || !p_traj || !src) return SL_ERR_ARG;
    if ((size_t)(T + 1) * (size_t)B > kNoAllocMaxSlots) return SL_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    int32_t *scratch = nullptr;
    if (noalloc_scratch(&scratch) != cudaSuccess) {
        cudaGetLastError();
        return SL_ERR_CUDA;
    }
    int32_t *tags = scratch, *last = scratch + kNoAllocMaxSlots, *err = scratch + 2 * kNoAllocMaxSlots;
    // the status word must start at zero; the kernel initialises every slot tag it reads
    if (cudaMemsetAsync(err, 0, sizeof(int32_t), st) != cudaSuccess) {
        cudaGetLastError();
        return SL_ERR_CUDA;
    }
    prepass_kernel<<<ceil_div(B, kPrepassThreads), kPrepassThreads, 0, st>>>(T, B, ops, p_traj, src, last, tags, err);
    int32_t h = 0;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return SL_ERR_CUDA;
    }
    return (sl_status)h;
}

