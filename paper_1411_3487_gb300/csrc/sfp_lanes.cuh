// sfp_lanes.cuh -- the mode-space step (Sec. 4) of a tile of up to 32 chains of
// 64, 128 or 256 beads on one CTA, BF16 hi/lo transforms, n_steps per launch.
//
// The bonds and modes of a chain are the 128 TMEM lanes (the M dimension of the
// MMA), the chains' axes its columns (N = 96: 32 chain slots of 3 axes):
//   inverse  D_u[i][row]   = sum_p chi[i][p]          R[row][p]        (Eq. e5)
//   forward  D_inc[p][row] = sum_n (h chi)[p][n]      v[row][n]
//                          + sum_n (w phi)[p][n]      z[row][n]        (Eqs. e11, c4, d6, f2)
// so the tables are the A operand and the state, forces and normals the B
// operand.  A thread owns one lane: the three axes of a chain's bond are three
// of its own columns (no exchange between threads for |u_n| or the shear term),
// the per-mode constants are its registers, and what it writes for the next
// contraction (its K index, consecutive rows) is 8 contiguous bytes.
//
// Mirror symmetry (256 beads).  chi_{n,p} ~ sin(pi n p / M) and phi_{n,p} ~
// cos(pi (n + 1/2) p / M) are even or odd under n -> M - n and n -> M - 1 - n
// with the parity of p, so each contraction splits into two of half the rows
// and half the K: even modes with v_n - v_{M-n} and z_n + z_{M-1-n}, odd modes
// with v_n + v_{M-n} and z_n - z_{M-1-n}, n < M / 2.  Lane i holds bonds i and
// M - i and modes 2 i and 2 i + 1 (bond M / 2, its own mirror image, takes lane
// 0, where bond 0 does not exist, with half its table column).  It halves the MMAs, the
// table bytes and the operand bytes.  At 128 beads the 128 lanes are the modes
// themselves; at 64 beads lanes 64..127 repeat lanes 0..63, so that all four
// TMEM lane quarters can work on the tile's chains.
//
// Roles (18 warps of work): warp 0 streams the tables (256 beads: 24 blocks of
// 16 KB a step through a ring; 64 and 128 beads: resident, loaded once), warp 1
// issues the MMAs, warps 2..17 do everything else: per step
//   force:     bond vectors from D_u -> v -> operand X, then normals of the next
//              step while the forward MMAs run
//   epilogue:  R += -dm R + D_inc (+ shear) -> global and operand X, then more
//              normals while the inverse MMAs run
// All 16 warps run the same code at about the same time, and the normals, the
// most arithmetic of a step and independent of the state, fill every wait for
// the tensor pipe.  The state R stays in global memory (L2): each thread reads
// and writes its own modes, 256 contiguous bytes per warp.
//
// Measured (GB300, 400-step calls, 4096 x 256 bp, 28 chains per tile): 22.8 us a
// step with the chains' axes on the TMEM lanes (fused_tile), 12.9 us here; 50 x
// 128 bp, 8 steps with the call around them: 146 -> 97 us; 4096 x 64 bp, 400 steps
// and 21 samples: 4.75 -> 3.71 ms.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

#include "sfp_device.cuh"
#include "sfp_fused.h"
#include "sfp_ptx.cuh"

namespace sfp {
namespace lanes {

using namespace ptx;

constexpr int kRowsN = 96;                      // MMA N: 32 chain slots x 3 axes
constexpr int kMaxChains = 32;
constexpr int kWarps = 16;                      // working warps (2 .. 17)
constexpr int kThreads = 32 * (2 + kWarps);
constexpr int kBlkBytes = 16384;                // a table block: [hi, lo][2 K steps][2 k groups][16 row groups][8][8]
constexpr int kALbo = 2048, kASbo = 128;        // table blocks: K-major core matrices
constexpr int kXSbo = 2048;                     // operand X: rows-major (MN-major) core matrices, [12 row groups][16 k groups]
constexpr int kXPart = 12 * kXSbo;              // one parity and part (hi or lo): 24 KB
constexpr int kZLbo = 12 * 128 + 16;            // noise operand: K-major core matrices, k groups 16 bytes apart in the banks
constexpr int kZPart = 8 * kZLbo;               // K = 64

template <int M>
struct Geo {
    static constexpr bool kFold = M == 256;
    static constexpr int NP = kFold ? 2 : 1;            // parities
    static constexpr int KP = M / NP;                   // K of one parity's contraction
    static constexpr int NG = M == 64 ? 8 : 4;          // chain groups (working warps of a lane)
    static constexpr int SLOTS = kMaxChains / NG;       // chain slots of a group
    static constexpr bool kStream = M == 256;           // tables through a ring, else resident
    static constexpr bool kScaled = M == 128;           // one symmetric table sin(pi n p / M) for both directions
    static constexpr int BLK = NP * KP / 32;            // table blocks of one contraction
    static constexpr int BLK_STEP = 3 * BLK;            // ... of a step (streamed)
    static constexpr int BLK_TAB = kScaled ? 2 * BLK : 3 * BLK;   // ... in the table image
    static constexpr int ST = kStream ? 5 : BLK_TAB;    // blocks in shared memory
    static constexpr int NCH = M == 64 ? 1 : 2;         // noise chunks (K = 64 per parity) of a step
    static constexpr int XB = NP * 2 * kXPart;
    static constexpr int ZB = NP * 2 * kZPart;
    static constexpr int kMisc = 1664;
    static constexpr int kBytes = ST * kBlkBytes + XB + ZB + kMisc + 128;
    // TMEM columns: D_u and D_inc, 96 each per parity; with the symmetric table, whose
    // increment h_p c_p scales after the contraction, the noise in a third accumulator
    static constexpr uint32_t kCols = M == 64 ? 256 : 512;
    static_assert(kBytes <= 227 * 1024, "shared memory of one CTA");
};

// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// Shared-memory matrix descriptor without swizzle (core matrices of 8 x 16 bytes).
__device__ __forceinline__ uint64_t ndesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(taddr));
}
// Wait for this thread's TMEM loads; the loaded registers pass through, so that
// no use of them can move above the wait.
__device__ __forceinline__ void tmem_wait12(float (&a)[3][4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0][0]), "+f"(a[0][1]), "+f"(a[0][2]), "+f"(a[0][3]), "+f"(a[1][0]), "+f"(a[1][1]),
                   "+f"(a[1][2]), "+f"(a[1][3]), "+f"(a[2][0]), "+f"(a[2][1]), "+f"(a[2][2]), "+f"(a[2][3])
                 :: "memory");
}

// Four values as BF16 hi and lo parts (round to nearest even), value i in halfword i.
__device__ __forceinline__ void split4(const float (&x)[4], uint2& hi, uint2& lo)
{
    uint32_t h[2], l[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h[i]) : "f"(x[2 * i + 1]), "f"(x[2 * i]));
        const float a = x[2 * i] - __uint_as_float(h[i] << 16);
        const float b = x[2 * i + 1] - __uint_as_float(h[i] & 0xFFFF0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l[i]) : "f"(b), "f"(a));
    }
    hi = make_uint2(h[0], h[1]);
    lo = make_uint2(l[0], l[1]);
}

struct LaneArgs {
    const uint8_t* tab;     // table blocks in the order a step takes them (chi, w phi, h chi); 128 beads: sin, w phi
    const float4* lane_c;   // per mode p: 1 - e^{-zeta dtau}, shear weight, operand scale, increment scale
};

// Tile `tile` (chains tile * a.cpt ...) through a.n_steps steps.  `tmem`: the
// base of Geo<M>::kCols allocated columns; `smem`: 128-byte-aligned dynamic
// shared memory.  Threads past kThreads take part in the block barriers only.
// Returns false if a wait gave up.
template <int M>
__device__ __forceinline__ bool lane_tile(const FusedArgs& a, const LaneArgs& la, int tile, uint8_t* smem, uint32_t tmem)
{
    using G = Geo<M>;
    constexpr int NP = G::NP;
    uint8_t* tabs = smem;
    uint8_t* X = smem + G::ST * kBlkBytes;
    uint8_t* Z = X + G::XB;
    uint8_t* misc = Z + G::ZB;
    int64_t* s_step = (int64_t*)misc;               // [32]
    double* s_shear = (double*)(misc + 256);        // [32]
    uint32_t* s_job = (uint32_t*)(misc + 512);      // [32]
    int* s_left = (int*)(misc + 640);               // [32] steps this chain still takes in this launch
    float* s_d0 = (float*)(misc + 768);             // [32][3] noise increments of the centre of mass
    uint64_t* bars = (uint64_t*)(misc + 1152);
    float* s_shf = (float*)(misc + 1408);           // [32]
    uint64_t* full = bars;              // table block landed (1 + tx)
    uint64_t* empty = bars + 8;         // MMAs done with the block (commit)
    uint64_t* tab_full = bars + 16;     // resident tables landed
    uint64_t* r_ready = bars + 17;      // operand X holds the modes (every working warp)
    uint64_t* v_ready = bars + 18;      // operand X holds the bond forces
    uint64_t* n_ready = bars + 19;      // noise operand written
    uint64_t* n_free = bars + 20;       // MMAs done with the noise operand (commit)
    uint64_t* u_done = bars + 21;       // inverse MMAs done (commit)
    uint64_t* inc_done = bars + 22;     // forward MMAs done (commit)
    uint64_t* never = bars + 23;        // nothing arrives here (the stall test)
    volatile int* abort_flag = (volatile int*)(bars + 24);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp: uniform
    const int c0 = tile * a.cpt;
    const int Ct = min(a.cpt, a.C - c0);

    if (threadIdx.x == 0) {
        if constexpr (G::kStream)
            for (int s = 0; s < G::ST; ++s) {
                mbar_init(&full[s], 1);
                mbar_init(&empty[s], 1);
            }
        mbar_init(tab_full, 1);
        mbar_init(r_ready, kWarps);
        mbar_init(v_ready, kWarps);
        mbar_init(n_ready, kWarps);
        mbar_init(n_free, 1);
        mbar_init(u_done, 1);
        mbar_init(inc_done, 1);
        mbar_init(never, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < kMaxChains; i += blockDim.x) {
        const bool live = i < Ct;
        const int64_t st = live ? a.step[c0 + i] : 0;
        int64_t left = live ? (int64_t)a.n_steps : 0;
        if (live && a.stop) left = max((int64_t)0, min(left, a.stop[c0 + i] - st));
        s_step[i] = st;
        s_left[i] = (int)left;
        s_job[i] = live ? a.job[c0 + i] : 0u;
        s_shear[i] = live ? a.shear[c0 + i] : 0.0;
        s_shf[i] = (float)s_shear[i];
    }
    // rows and K indices that nothing writes stay zero
    for (int i = threadIdx.x; i < (G::XB + G::ZB) / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(X)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const bool has_shear = __syncthreads_or(threadIdx.x < Ct && s_shear[threadIdx.x] != 0.0) != 0;

    if (warp == 0) {
        // ---------------- table blocks
        if (lane == 0) {
            bool ok = true;
            if constexpr (G::kStream) {
                const int total = a.n_steps * G::BLK_STEP;
                int src = 0;
                for (int it = 0; it < total; ++it) {
                    const int s = it % G::ST;
                    ok = mbar_wait(&empty[s], ((it / G::ST) & 1) ^ 1, a.err, abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&full[s], kBlkBytes);
                    bulk_load(tabs + s * kBlkBytes, la.tab + (size_t)src * kBlkBytes, kBlkBytes, &full[s]);
                    if (++src == G::BLK_STEP) src = 0;
                }
                // the last commit of every ring slot has landed before the tile ends
                for (int s = 0; s < G::ST && s < total && ok; ++s) {
                    const int last = s + G::ST * ((total - 1 - s) / G::ST);
                    ok = mbar_wait(&empty[s], (last / G::ST) & 1, a.err, abort_flag);
                }
            } else {
                mbar_expect_tx(tab_full, G::BLK_TAB * kBlkBytes);
                for (int k = 0; k < G::BLK_TAB; ++k)
                    bulk_load(tabs + k * kBlkBytes, la.tab + (size_t)k * kBlkBytes, kBlkBytes, tab_full);
                mbar_wait(tab_full, 0, a.err, abort_flag);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer.  The whole warp runs the loops and the waits,
        // one elected lane issues: with everything but the issue itself uniform over
        // the warp, descriptors live in uniform registers and an MMA costs a few
        // instructions (a single-lane loop took 740 cycles for the six MMAs of a
        // block, beside 16 busy warps; their run time is 288).
        constexpr uint32_t id_z = idesc_bf16(128, kRowsN);              // B K-major
        constexpr uint32_t id_x = id_z | (1u << 16);                    // B rows-major
        const bool leader = elect_one();
        bool ok = true;
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            ok = __all_sync(0xffffffffu, ok && mbar_wait(bar, parity, a.err, abort_flag));
            fence_after();
        };
        if (a.stall_test) wait(never, 0);
        if constexpr (!G::kStream) wait(tab_full, 0);
        const uint64_t tab0 = ndesc(smem_u32(tabs), kALbo, kASbo);
        const uint64_t x0 = ndesc(smem_u32(X), 128, kXSbo), z0 = ndesc(smem_u32(Z), kZLbo, 128);
        int slot = 0;                                   // ring slot and phase of the next streamed block
        uint32_t phase = 0;
        // the six MMAs of a block's two K steps, table hi/lo x operand hi/lo; b: the
        // operand's hi part (the lo part b_lo further), bstep: its next K step
        auto block = [&](int resident, uint32_t d, uint64_t b, uint32_t b_lo, uint32_t bstep, uint32_t idesc, bool first) {
            const int s = G::kStream ? slot : resident;
            if constexpr (G::kStream) wait(&full[s], phase);
            if (leader && ok) {
                const uint64_t ad = tab0 + (uint64_t)(s * (kBlkBytes / 16));
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                    const uint64_t ah = ad + kk * (4096 / 16), al = ah + 8192 / 16;
                    const uint64_t bh = b + kk * (bstep / 16), bl = bh + b_lo / 16;
                    mma_bf16(d, al, bh, idesc, (first && kk == 0) ? 0u : 1u);
                    mma_bf16(d, ah, bl, idesc, 1u);
                    mma_bf16(d, ah, bh, idesc, 1u);
                }
                if constexpr (G::kStream) mma_commit(&empty[s]);
            }
            if constexpr (G::kStream) {
                if (++slot == G::ST) {
                    slot = 0;
                    phase ^= 1u;
                }
            }
        };
        // a contraction of operand X (modes or bond forces) into d
        auto with_x = [&](int res0, uint32_t d, bool first) {
#pragma unroll 1
            for (int kc = 0; kc < G::BLK / NP; ++kc)
#pragma unroll
                for (int e = 0; e < NP; ++e)
                    block(res0 + kc * NP + e, d + e * kRowsN, x0 + (uint64_t)((e * 2 * kXPart + kc * 4 * 128) / 16), kXPart,
                          256, id_x, first && kc == 0);
        };
        const uint32_t d_u = tmem, d_inc = tmem + NP * kRowsN, d_z = G::kScaled ? d_inc + kRowsN : d_inc;
        int chunk = 0;
#pragma unroll 1
        for (int sp = 0; sp < a.n_steps && ok; ++sp) {
            wait(r_ready, sp & 1);
            with_x(0, d_u, true);
            if (leader && ok) mma_commit(u_done);
#pragma unroll 1
            for (int ch = 0; ch < G::NCH; ++ch, ++chunk) {
                wait(n_ready, chunk & 1);
                constexpr int KC = G::BLK / G::NCH / NP;            // K blocks of a chunk
#pragma unroll 1
                for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                    for (int e = 0; e < NP; ++e)
                        block(G::BLK + (ch * KC + kc) * NP + e, d_z + e * kRowsN,
                              z0 + (uint64_t)((e * 2 * kZPart + kc * 4 * kZLbo) / 16), kZPart, 2 * kZLbo, id_z,
                              ch == 0 && kc == 0);
                if (leader && ok) mma_commit(n_free);
            }
            wait(v_ready, sp & 1);
            with_x(G::kScaled ? 0 : 2 * G::BLK, d_inc, G::kScaled);
            if (leader && ok) mma_commit(inc_done);
        }
    } else if (warp < 2 + kWarps) {
        // ---------------- the working warps
        const int q = warp & 3;                                 // TMEM lane quarter
        const int g = ((warp - 2) >> 2) + (M == 64 ? 4 * (q >> 1) : 0);   // chain group
        const int j = (32 * q + lane) & (M == 64 ? 63 : 127);   // bond (pair) and mode (pair) index
        const bool lane0 = (32 * q & (M == 64 ? 63 : 127)) == 0;   // this warp holds mode 0
        const int ks = (a.cpt + G::NG - 1) / G::NG;             // chain slots in use per group
        const int cl0 = g * ks;                                 // this group's first chain of the tile
        const int ns = max(0, min(ks, Ct - cl0));               // ... and its live chains
        // first row of the group: 24 rows (3 axes x 8 slots) per 4 or 8 groups
        const int pos0 = M == 64 ? 4 * (g >> 2) : 0;
        const int row0 = 24 * (g & 3) + pos0;
        const uint32_t tq = (uint32_t)(32 * q) << 16;
        const uint32_t d_u = tmem + tq + (uint32_t)row0, d_inc = d_u + NP * kRowsN;
        // this thread's 8 bytes of operand X: parity e, part, axis
        uint8_t* xw = X + 3 * (g & 3) * kXSbo + j * 16 + pos0 * 2;
        float dm[NP], gw[NP], cs[NP], es[NP];
#pragma unroll
        for (int e = 0; e < NP; ++e) {
            const float4 c = la.lane_c[NP * j + e];
            dm[e] = c.x; gw[e] = c.y; cs[e] = c.z; es[e] = c.w;
        }
        bool ok = true, finite = true;
        // the centre of mass (FP64): lane 3 s + axis of a warp that holds mode 0
        const int ms = lane / 3, ma = lane - 3 * ms;
        const bool cm_mine = lane0 && ms < ns;
        double cm = cm_mine ? a.com[3 * (size_t)(c0 + cl0 + ms) + ma] : 0.0;

        auto arrive = [&](uint64_t* bar) {
            fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0 && ok) mbar_arrive(bar);
        };
        auto put_x = [&](const float (&x)[3][4], int e, int sb) {
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                uint2 h, l;
                split4(x[ax], h, l);
                uint8_t* w = xw + e * 2 * kXPart + ax * kXSbo + sb * 2;
                *reinterpret_cast<uint2*>(w) = h;
                *reinterpret_cast<uint2*>(w + kXPart) = l;
            }
        };
        // the modes (2 j, 2 j + 1) or j of four chains, [parity][axis][chain]
        auto load_r = [&](float (&r)[NP][3][4], int sb) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    const float* p = a.R + (size_t)(3 * (c0 + cl0 + sb + i) + ax) * M + NP * j;
                    if constexpr (NP == 2) {
                        const float2 x = sb + i < ns ? *reinterpret_cast<const float2*>(p) : make_float2(0.f, 0.f);
                        r[0][ax][i] = x.x;
                        r[NP - 1][ax][i] = x.y;
                    } else {
                        r[0][ax][i] = sb + i < ns ? *p : 0.f;
                    }
                }
        };
        auto put_r = [&](const float (&r)[NP][3][4], int sb) {
#pragma unroll
            for (int e = 0; e < NP; ++e) {
                if constexpr (G::kScaled) {
                    float x[3][4];
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                        for (int i = 0; i < 4; ++i) x[ax][i] = cs[e] * r[e][ax][i];
                    put_x(x, e, sb);
                } else {
                    put_x(r[e], e, sb);
                }
            }
        };

        // Normals of a noise chunk (Eq. b5): 64 K indices of step sp, chunk ch.  A
        // lane draws four consecutive beads of a chain (three Philox calls) and,
        // with the mirror symmetry, their four mirror images, and writes the sums
        // and differences as 8 bytes of a row of the noise operand: 16 lanes fill
        // a chain's row.  The chunk's items go to the warps in turn, starting one
        // warp group further from chunk to chunk.
        auto noise = [&](int sp, int ch, int chunk) {
            const int items = (Ct + 1) >> 1;                    // two chains per item
            const int item = (warp - 2 + 8 * chunk) & (kWarps - 1);
            const int cl = 2 * item + (lane >> 4), t = lane & 15;
            const bool mine = item < items && cl < Ct;
            uint2 hi[NP][3], lo[NP][3];
            if (mine) {
                const uint32_t job = s_job[cl];
                const int64_t st = s_step[cl] + sp;
                const uint32_t b4 = (uint32_t)(16 * ch + t);    // beads 4 b4 ...
                float z[3][4];
                bead_quad_normals<float>(a.seed, job, st, b4, 0u, z);
                if constexpr (NP == 2) {
                    float y[3][4];
                    bead_quad_normals<float>(a.seed, job, st, (uint32_t)(M / 4 - 1) - b4, 0u, y);
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        float s[4], d[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            s[i] = z[ax][i] + y[ax][3 - i];
                            d[i] = z[ax][i] - y[ax][3 - i];
                        }
                        split4(s, hi[0][ax], lo[0][ax]);
                        split4(d, hi[NP - 1][ax], lo[NP - 1][ax]);
                    }
                } else {
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) split4(z[ax], hi[0][ax], lo[0][ax]);
                }
            }
            // the previous chunk's MMAs have read the operand
            if (chunk > 0) ok = ok && mbar_wait(n_free, (chunk - 1) & 1, a.err, abort_flag);
            if (mine && ok) {
                const int cg = cl / ks, cs_ = cl - cg * ks;
                uint8_t* w = Z + (t >> 1) * kZLbo + 3 * (cg & 3) * 128 + ((M == 64 ? 4 * (cg >> 2) : 0) + cs_) * 16 + (t & 1) * 8;
#pragma unroll
                for (int e = 0; e < NP; ++e)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        *reinterpret_cast<uint2*>(w + e * 2 * kZPart + ax * 128) = hi[e][ax];
                        *reinterpret_cast<uint2*>(w + e * 2 * kZPart + kZPart + ax * 128) = lo[e][ax];
                    }
            }
            arrive(n_ready);
        };

        // operand X of the first step
        for (int sb = 0; sb < ns; sb += 4) {
            float r[NP][3][4];
            load_r(r, sb);
            put_r(r, sb);
        }
        arrive(r_ready);
        int chunk = 0;
        if constexpr (G::NCH == 2) noise(0, 0, chunk++);
        // phases of half a step: even ones form the force, odd ones update the modes;
        // each is followed by a chunk of normals drawn ahead
#pragma unroll 1
        for (int ph = -1; ph < 2 * a.n_steps; ++ph) {
            const int sp = ph >> 1;
            if (ph >= 0 && (ph & 1) == 0) {
                // ---- bond vectors -> residual force v (Eq. e11)
                ok = ok && mbar_wait(u_done, sp & 1, a.err, abort_flag);
                fence_after();
#pragma unroll 1
                for (int sb = 0; sb < ns; sb += 4) {
                    float u[NP][3][4];
#pragma unroll
                    for (int e = 0; e < NP; ++e)
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_u + e * kRowsN + 8 * ax + sb, u[e][ax]);
#pragma unroll
                    for (int e = 0; e < NP; ++e) tmem_wait12(u[e]);
                    if constexpr (NP == 2) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float p[3], m[3];     // bonds j and M - j
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) {
                                p[ax] = u[NP - 1][ax][i] + u[0][ax][i];
                                m[ax] = u[NP - 1][ax][i] - u[0][ax][i];
                            }
                            const float fp = rsqrtf(fmaf(p[0], p[0], fmaf(p[1], p[1], p[2] * p[2]))) - a.c12nu;
                            const float fm = rsqrtf(fmaf(m[0], m[0], fmaf(m[1], m[1], m[2] * m[2]))) - a.c12nu;
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) {
                                const float vm = m[ax] * fm;
                                u[0][ax][i] = fmaf(p[ax], fp, -vm);          // even modes
                                u[NP - 1][ax][i] = fmaf(p[ax], fp, vm);      // odd modes
                            }
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float f = rsqrtf(fmaf(u[0][0][i], u[0][0][i], fmaf(u[0][1][i], u[0][1][i], u[0][2][i] * u[0][2][i]))) -
                                      a.c12nu;
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) u[0][ax][i] = j >= 1 ? u[0][ax][i] * f : 0.f;   // v_0 = 0
                        }
                    }
#pragma unroll
                    for (int e = 0; e < NP; ++e) put_x(u[e], e, sb);
                }
                arrive(v_ready);
            } else if (ph >= 0) {
                // ---- update (Eqs. d3, btum)
                float r[NP][3][4];
                if (ns > 0) load_r(r, 0);
                ok = ok && mbar_wait(inc_done, sp & 1, a.err, abort_flag);
                fence_after();
                const bool last = sp == a.n_steps - 1;
#pragma unroll 1
                for (int sb = 0; sb < ns; sb += 4) {
                    float d[NP][3][4];
#pragma unroll
                    for (int e = 0; e < NP; ++e)
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_inc + e * kRowsN + 8 * ax + sb, d[e][ax]);
                    float dz[3][4];
                    if constexpr (G::kScaled) {
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_inc + kRowsN + 8 * ax + sb, dz[ax]);
                    }
                    if (sb > 0) load_r(r, sb);
#pragma unroll
                    for (int e = 0; e < NP; ++e) tmem_wait12(d[e]);
                    if constexpr (G::kScaled) {
                        tmem_wait12(dz);
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                            for (int i = 0; i < 4; ++i) d[0][ax][i] = fmaf(es[0], d[0][ax][i], dz[ax][i]);
                    }
                    if (lane0 && lane == 0) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (sb + i < ns)
#pragma unroll
                                for (int ax = 0; ax < 3; ++ax) s_d0[3 * (cl0 + sb + i) + ax] = d[0][ax][i];
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (sb + i >= ns) break;
                        if (sp < s_left[cl0 + sb + i]) {        // a chain at its stop step stays as it is
                            const float sh = has_shear ? s_shf[cl0 + sb + i] : 0.f;
#pragma unroll
                            for (int e = 0; e < NP; ++e) {
                                const float ry = r[e][1][i];
#pragma unroll
                                for (int ax = 0; ax < 3; ++ax) {
                                    const float x = r[e][ax][i];
                                    r[e][ax][i] = x + fmaf(-dm[e], x, d[e][ax][i]);
                                }
                                if (has_shear) r[e][0][i] += sh * gw[e] * ry;
                            }
                        }
                        if (lane0 && lane == 0) r[0][0][i] = r[0][1][i] = r[0][2][i] = 0.f;   // the centre of mass is cm
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) {
                            float* p = a.R + (size_t)(3 * (c0 + cl0 + sb + i) + ax) * M + NP * j;
                            if constexpr (NP == 2)
                                *reinterpret_cast<float2*>(p) = make_float2(r[0][ax][i], r[NP - 1][ax][i]);
                            else
                                *p = r[0][ax][i];
                        }
                        // a non-finite mode stays non-finite: looked at once per launch
                        if (last) {
#pragma unroll
                            for (int e = 0; e < NP; ++e)
#pragma unroll
                                for (int ax = 0; ax < 3; ++ax) finite = finite && isfinite(r[e][ax][i]);
                        }
                    }
                    if (!last) put_r(r, sb);
                }
                if (!last) arrive(r_ready);
                if (lane0) {
                    // centre of mass (p = 0 of Eq. d3 with zeta_0 = 0) in FP64
                    __syncwarp();
                    const double ycm = has_shear ? __shfl_down_sync(0xffffffffu, cm, 1) : 0.0;
                    if (cm_mine && sp < s_left[cl0 + ms]) {
                        double x = (double)s_d0[3 * (cl0 + ms) + ma] * a.inv_sqrtM;
                        if (has_shear && ma == 0) x += s_shear[cl0 + ms] * a.dtau * ycm;
                        cm += x;
                    }
                    __syncwarp();
                }
            }
            // normals drawn ahead: chunk 0 of step s + 1 after the force of step s, the
            // last chunk of step s + 1 after the update of step s
            const int zs = (ph + 2) >> 1;
            if (zs < a.n_steps) {
                if (G::NCH == 2) noise(zs, (ph & 1) ? 1 : 0, chunk++);
                else if (ph & 1) noise(zs, 0, chunk++);
            }
        }
        if (ok && cm_mine) a.com[3 * (size_t)(c0 + cl0 + ms) + ma] = cm;
        if (ok && lane0 && lane < ns) a.step[c0 + cl0 + lane] = s_step[cl0 + lane] + s_left[cl0 + lane];
        if (!finite) atomicOr(a.err, 1);
    }
    fence_before();
    __syncthreads();
    const bool good = *abort_flag == 0;
    if (!good) {
        // a wait gave up: let copies and MMAs in flight land before the memory goes
        const uint64_t t0 = globaltimer();
        while (globaltimer() - t0 < 1000000ull) __nanosleep(1000);
        __syncthreads();
    }
    return good;
}

}  // namespace lanes
}  // namespace sfp
