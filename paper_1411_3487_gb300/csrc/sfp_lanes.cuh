// sfp_lanes.cuh -- the mode-space step (Sec. 4) of a tile of up to 32 chains of
// 64, 128 or 256 beads on one CTA, or up to 24 of 512 beads on a cluster of two,
// BF16 hi/lo transforms, n_steps per launch.
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
// Roles (20 warps): warp 0 streams the tables (256 beads: 24 pairs of blocks, 16 KB each, a step
// through a ring; 64 and 128 beads: resident, loaded once); warp 1 issues the MMAs
// (256 beads: of the even modes, warp 18 of the odd ones, whose accumulators are
// others); warps 2..9 (two per TMEM lane quarter) form the force, D_u -> v -> operand
// X, and update the modes, R += -dm R + D_inc (+ shear) -> operand X; warps 10..17
// draw the normals, the most arithmetic of a step and independent of the state, into
// the two buffers of the noise operand; warp 19 keeps the FP64 centre of mass.  The
// chain of a step, inverse MMAs - force - forward MMAs - update, then leaves most
// issue slots to the normals.  The state stays in TMEM for the launch; at 256 beads
// three of eight batches of chains find no room there and live in global memory (L2),
// read and written by the thread that owns the modes.
//
// What bounds it (256 beads, 28 chains): the chain of a step, 5.3 us with one chain per
// tile (inverse and forward MMAs 3000 cycles each, force, update and four hand-overs),
// stretched by what shares the SM with it: 42.8 K warp instructions a step at 2.5 a
// cycle, the normals' more than half.  Neither pipe is full: a capture of three steps
// shows the issue slots 46 % busy and the tensor pipe 30 % active.  State and D live in
// 504 of the 512 TMEM columns.
// 512 beads (a cluster of two CTAs): the parities of the mirror symmetry are 256 modes
// each, two row tiles of 128, and CTA rank r takes parity r, so that its operand, its
// share of the state and its table stream are what one CTA holds at 256 beads.  Bonds are
// sums over both parities: after the inverse MMAs each CTA sends the other the parts of
// D_u of that one's 128 bond lanes (32 KB a step each way), works out both parities' force
// operand for its own lanes, keeps one and stores the other in its peer's operand X.  The
// normals are drawn once: each CTA draws every second chunk and writes the sums to the
// even modes' CTA and the differences to the other.  All of it goes by st.async, which
// counts bytes on the reader's mbarrier, so that nobody waits for the stores (with plain
// remote stores and remote arrivals: 197 us a step at 16384 chains instead of 175 then).  Half
// of the noise chunks come after the forward MMAs, so that their way between the CTAs
// passes behind those.  The step is bound by its chain, 10 us of 14.5 at 24 chains: inverse
// and forward MMAs 5 us with their waits for 768 KB of tables (64 KB under way in the
// ring, what operands and buffers leave), two exchanges, force, update.
//
// Measured (GB300, us a step in a 400-step call, the four-role kernel of sfp_fused.cu
// before -> here): 4096 x 256 bp 22.7 -> 8.9, 8 x 256 bp 19.1 -> 5.2, 4096 x 128 bp
// 10.3 -> 4.3, 50 x 128 bp 9.5 -> 2.7, 4096 x 64 bp 7.3 -> 2.4, 8 x 64 bp 5.9 -> 1.5; 16384 x 512 bp 289 ->
// 132 (here 1000 x 512 bp take 11.9, one chain 10.0).
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

#include "sfp_device.cuh"
#include "sfp_fused.h"
#include "sfp_ptx.cuh"

namespace sfp {
namespace lanes {

using namespace ptx;

constexpr int kMaxSlots = 32;                   // chain slots of the shared-memory arrays
constexpr int kWork = 8, kNoise = 8;            // force / update warps (2 .. 9), noise warps (10 .. 17)
constexpr int kThreads = 32 * (4 + kWork + kNoise);
constexpr int kBlkBytes = 8192;                 // a table block (one K step of 16): [hi, lo][2 k groups][16 row groups][8][8]
constexpr int kALbo = 2048, kASbo = 128;        // table blocks: K-major core matrices

// Rows of N: four chains (batch b = chain / 4 of the tile) hold rows 24 (b / 2) +
// 8 axis + 4 (b & 1) + chain % 4 (Geo::pair, Geo::half), so that a thread's four values of an axis are 8
// contiguous bytes of operand X.
template <int M>
struct Geo {
    static constexpr bool kPair = M == 512;             // a tile on a cluster of two CTAs, a parity each
    static constexpr bool kFold = M >= 256;             // mirror symmetry
    static constexpr int NP = kFold ? 2 : 1;            // accumulators: the parities, or the two row tiles of this CTA's parity
    static constexpr int KP = kFold ? M / 2 : M;        // K of a contraction
    static constexpr int ROWS = kPair ? 80 : 96;        // MMA N at most: chain slots x 3 axes (72 of 80 used)
    static constexpr int GROUPS = kPair ? 9 : 12;       // row groups of 8
    static constexpr int kMaxChains = 8 * GROUPS / 3;
    // Where batch b's rows lie: rows 24 pair + 8 axis + 4 half + chain.  A pair of CTAs puts
    // batches 0 | 2 and 1 | 3 side by side, which one warp works on, so that what it
    // stores in the other CTA is 16 bytes a lane.
    __device__ static constexpr int pair(int b) { return kPair && b < 4 ? b & 1 : b >> 1; }
    __device__ static constexpr int half(int b) { return kPair && b < 4 ? b >> 1 : b & 1; }
    // pairs of batches that n batches take
    __device__ static constexpr int pairs(int n) { return kPair ? (n <= 1 ? 1 : n <= 4 ? 2 : 3) : (n + 1) >> 1; }
    static constexpr bool kStream = M >= 256;           // tables through a ring, else resident
    static constexpr bool kScaled = M == 128;           // one symmetric table sin(pi n p / M) for both directions
    static constexpr int ZK = kPair ? 64 : 32;          // K of a noise chunk
    static constexpr int NCH = KP / ZK;                 // noise chunks of a step
    static constexpr int BLK = NP * KP / 16;            // table blocks of one contraction
    static constexpr int BLK_STEP = 3 * BLK;            // ... of a step (streamed)
    static constexpr int BLK_TAB = kScaled ? 2 * BLK : 3 * BLK;   // ... in the table image (of one CTA of a pair)
    // blocks in shared memory: all, or a ring, whose slots hold the blocks of both
    // accumulators for the same K indices, one copy of 16 KB
    static constexpr int ST = kPair ? 8 : kStream ? 10 : BLK_TAB;
    static constexpr int SLOTS = ST / NP;
    static_assert(!kStream || ST % NP == 0, "whole slots");
    static constexpr int PAR = kPair ? 1 : NP;          // parities whose operands this CTA holds
    // operand X: rows-major (MN-major) core matrices, [GROUPS][KP / 8]
    static constexpr int XSBO = KP * 16, XPART = GROUPS * XSBO, XB = PAR * 2 * XPART;
    // a buffer of the noise operand: K-major core matrices, k groups 32 bytes apart in the banks
    static constexpr int ZLBO = ROWS / 8 * 128 + 32, ZPART = ZK / 8 * ZLBO, ZB = PAR * 2 * ZPART;
    static constexpr int UB = kPair ? 2 * GROUPS * 2048 : 0;   // bond vectors from the other CTA, [batch][axis][128 lanes][4 chains]
    static constexpr int kMisc = 1664;
    static constexpr int kBytes = ST * kBlkBytes + XB + 2 * ZB + UB + kMisc + 128;
    // TMEM columns: D_u and D_inc, ROWS each per accumulator; with the symmetric table,
    // whose increment h_p c_p scales after the contraction, the noise in a third one;
    // then the state R of the first TB batches
    static constexpr uint32_t kCols = 512;
    static constexpr int kRCol = (2 * NP + (kScaled ? 1 : 0)) * ROWS;
    static constexpr int TB = (512 - kRCol) / (12 * NP) < 8 ? (512 - kRCol) / (12 * NP) : 8;
    static_assert(kBytes <= 227 * 1024, "shared memory of one CTA");
    static_assert(!kPair || 4 * TB >= kMaxChains, "a pair's whole state in TMEM");
};

// Stores to the other CTA's shared memory that count as transaction bytes of its
// mbarrier `bar` (cluster addresses): the writer neither waits for them nor arrives.
// A warp's 16 bytes a lane side by side take 31 cycles, 8 bytes a lane 16 bytes apart 69.
__device__ __forceinline__ void st_peer16(uint32_t addr, uint4 v, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
                 ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_peer8(uint32_t addr, uint2 v, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1,%2}, [%3];"
                 ::"r"(addr), "r"(v.x), "r"(v.y), "r"(bar) : "memory");
}

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

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const float (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
                 ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Two values as BF16 hi and lo parts (round to nearest even), value i in halfword i.
__device__ __forceinline__ void split2(f32x2 x, uint32_t& hi, uint32_t& lo)
{
    float a, b;
    unpack2(x, a, b);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
    unpack2(sub2(x, pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xFFFF0000u))), a, b);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(b), "f"(a));
}
__device__ __forceinline__ void split4(const float (&x)[4], uint2& hi, uint2& lo)
{
    split2(pack2(x[0], x[1]), hi.x, lo.x);
    split2(pack2(x[2], x[3]), hi.y, lo.y);
}

// 1/|u| of two bonds; |u|^2 of a bond that exists is far from the denormals.
__device__ __forceinline__ f32x2 rsqrt2(f32x2 t)
{
    float a, b;
    unpack2(t, a, b);
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(a));
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(b));
    return pack2(a, b);
}

struct LaneArgs {
    const uint8_t* tab;     // table blocks chi, w phi, h chi (128 beads: sin, w phi), K blocks in order, even modes first
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
    uint8_t* U = Z + 2 * G::ZB;
    uint8_t* misc = U + G::UB;
    int64_t* s_step = (int64_t*)misc;               // [32]
    double* s_shear = (double*)(misc + 256);        // [32]
    uint32_t* s_job = (uint32_t*)(misc + 512);      // [32]
    int* s_left = (int*)(misc + 640);               // [32] steps this chain still takes in this launch
    float* s_d0 = (float*)(misc + 768);             // [3][32] noise increments of the centre of mass
    uint64_t* bars = (uint64_t*)(misc + 1152);
    float* s_shf = (float*)(misc + 1456);           // [32]
    uint64_t* full = bars;              // ring slot: table blocks landed (1 + tx)
    uint64_t* empty = bars + 12;        // ... MMAs done with it (a commit per accumulator)
    uint64_t* tab_full = bars + 24;     // resident tables landed
    uint64_t* r_ready = bars + 25;      // operand X holds the modes, D_inc has been read (every work warp)
    uint64_t* v_ready = bars + 26;      // operand X holds the bond forces (every work warp; warp 19: s_d0 has been read; pair: + tx)
    uint64_t* n_ready = bars + 27;      // noise buffer b written (every noise warp)
    uint64_t* n_free = bars + 29;       // MMAs done with noise buffer b (a commit per parity)
    uint64_t* u_done = bars + 31;       // inverse MMAs done (a commit per parity)
    uint64_t* inc_done = bars + 32;     // noise and forward MMAs done (a commit per parity)
    uint64_t* never = bars + 33;        // nothing arrives here (the stall test)
    uint64_t* u_in = bars + 34;         // pair: the other CTA's bond vectors are in U (1 + tx)
    volatile int* abort_flag = (volatile int*)(bars + 35);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp: uniform
    const int c0 = tile * a.cpt;
    const int Ct = min(a.cpt, a.C - c0);
    const uint32_t rank = G::kPair ? cluster_rank() : 0u;
    // an address of this CTA's shared memory in the other CTA of the pair
    auto peer = [&](const void* p) { return mapa(smem_u32(p), rank ^ 1u); };

    if (threadIdx.x == 0) {
        if constexpr (G::kStream)
            for (int s = 0; s < G::SLOTS; ++s) {
                mbar_init(&full[s], 1);
                mbar_init(&empty[s], NP);
            }
        mbar_init(tab_full, 1);
        mbar_init(r_ready, kWork);
        mbar_init(v_ready, kWork + 1);
        mbar_init(u_in, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&n_ready[b], G::kPair && b != (int)rank ? 1 : kNoise);    // a pair's other buffer: transaction bytes
            mbar_init(&n_free[b], (G::kPair ? 2 : 1) * NP);
        }
        mbar_init(u_done, NP);
        mbar_init(inc_done, NP);
        mbar_init(never, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < kMaxSlots; i += blockDim.x) {
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
    for (int i = threadIdx.x; i < (G::XB + 2 * G::ZB) / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(X)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
    fence_before();
    if constexpr (G::kPair) cluster_sync();     // both CTAs' barriers are initialised
    else __syncthreads();
    fence_after();
    const bool has_shear = __syncthreads_or(threadIdx.x < Ct && s_shear[threadIdx.x] != 0.0) != 0;
    // no chain of the tile is sheared or reaches its stop step in this launch
    const bool steady = __syncthreads_and(!has_shear && (threadIdx.x >= Ct || s_left[threadIdx.x] == a.n_steps)) != 0;

    if (warp == 0) {
        const uint8_t* tab = la.tab + (G::kPair ? rank * (uint32_t)(G::BLK_TAB * kBlkBytes) : 0u);
        // ---------------- table blocks (the whole warp runs the loop, one lane issues:
        // see the MMA issuer)
        const bool leader = elect_one();
        if constexpr (G::kStream) {
            constexpr int STEP = G::BLK_STEP / NP, ONE = G::BLK / NP;     // slots of a step, of a contraction
            const int total = a.n_steps * STEP;
            bool ok = true;
            int s = 0, src = 0;
            uint32_t phase = 1;
#pragma unroll 1
            for (int it = 0; it < total; ++it) {
                ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], phase, a.err, abort_flag));
                if (!ok) break;
                if (leader) {
                    mbar_expect_tx(&full[s], NP * kBlkBytes);
                    // a pair's step takes the second half of w phi after h chi
                    const int k = !G::kPair || src < 3 * ONE / 2 ? src : src < 5 * ONE / 2 ? src + ONE / 2 : src - ONE;
                    bulk_load(tabs + s * (NP * kBlkBytes), tab + k * (NP * kBlkBytes), NP * kBlkBytes, &full[s]);
                }
                if (++src == STEP) src = 0;
                if (++s == G::SLOTS) {
                    s = 0;
                    phase ^= 1u;
                }
            }
            // the last commit of every ring slot has landed before the tile ends
            for (int k = 0; k < G::SLOTS && k < total && ok; ++k) {
                const int last = k + G::SLOTS * ((total - 1 - k) / G::SLOTS);
                ok = mbar_wait(&empty[k], (last / G::SLOTS) & 1, a.err, abort_flag);
            }
        } else {
            if (leader) {
                mbar_expect_tx(tab_full, G::BLK_TAB * kBlkBytes);
                for (int k = 0; k < G::BLK_TAB; ++k)
                    bulk_load(tabs + k * kBlkBytes, tab + k * kBlkBytes, kBlkBytes, tab_full);
            }
            mbar_wait(tab_full, 0, a.err, abort_flag);
        }
    } else if (warp == 1 || (NP == 2 && warp == 18)) {
        const int e = warp == 1 ? 0 : NP - 1;           // this warp's accumulator
        // ---------------- MMA issuer.  The whole warp runs the loops and the waits,
        // one elected lane issues: with everything but the issue itself uniform over
        // the warp, descriptors live in uniform registers and an MMA costs a few
        // instructions (a single-lane loop took 740 cycles for the six MMAs of a
        // block, beside 16 busy warps; their run time is 288).
        // N: the rows of the batches in use (24 per two batches), a multiple of 16
        const uint32_t id_z = idesc_bf16(128, (24 * G::pairs((Ct + 3) >> 2) + 15) & ~15);       // B K-major
        const uint32_t id_x = id_z | (1u << 16);                                        // B rows-major
        const bool leader = elect_one();
        bool ok = true;
        // peer: the barrier counts stores of the other CTA's threads into this CTA's shared
        // memory; a proxy fence on this side, for this CTA's shared memory, orders the MMAs
        // after them (one for every state space took 1200 cycles, six times a step)
        auto wait = [&](uint64_t* bar, uint32_t parity, bool peer) {
            if (G::kPair && peer) {
                ok = __all_sync(0xffffffffu, ok && mbar_wait_cl(bar, parity, a.err, abort_flag));
                fence_proxy_async();
            } else {
                ok = __all_sync(0xffffffffu, ok && mbar_wait(bar, parity, a.err, abort_flag));
            }
            fence_after();
        };
        if (a.stall_test) wait(never, 0, false);
        if constexpr (!G::kStream) wait(tab_full, 0, false);
        const uint64_t tab0 = ndesc(smem_u32(tabs), kALbo, kASbo);
        const int ep = G::kPair ? 0 : e;                // operands: of this parity, or of the CTA's
        const uint32_t z_bytes = (uint32_t)(G::ZK * 12 * Ct);       // a chunk of the other CTA: K x 3 axes x (hi, lo)
        const uint64_t x0 = ndesc(smem_u32(X) + ep * 2 * G::XPART, 128, G::XSBO), z0 = ndesc(smem_u32(Z) + ep * 2 * G::ZPART, G::ZLBO, 128);
        int slot = 0;                                   // ring slot and phase of the next streamed block
        uint32_t phase = 0;
        // the three MMAs of a block, table hi/lo x operand hi/lo; b: the operand's hi
        // part (the lo part b_lo further)
        auto block = [&](int resident, uint32_t d, uint64_t b, uint32_t b_lo, uint32_t idesc, bool first) {
            const int s = G::kStream ? NP * slot + e : resident;
            if constexpr (G::kStream) {
                ok = __all_sync(0xffffffffu, ok && mbar_wait(&full[slot], phase, a.err, abort_flag));
                fence_after();
            }
            if (leader && ok) {
                const uint64_t ah = tab0 + (uint64_t)(s * (kBlkBytes / 16)), al = ah + kBlkBytes / 32, bl = b + b_lo / 16;
                mma_bf16(d, al, b, idesc, first ? 0u : 1u);
                mma_bf16(d, ah, bl, idesc, 1u);
                mma_bf16(d, ah, b, idesc, 1u);
                if constexpr (G::kStream) mma_commit(&empty[slot]);
            }
            if constexpr (G::kStream) {
                if (++slot == G::SLOTS) {
                    slot = 0;
                    phase ^= 1u;
                }
            }
        };
        // unrolled where slots are constants; at 256 beads the loops stay small, for the
        // instruction cache (32 KB of code in the four roles' loops: 10.3 us a step, 9.1 below that)
        constexpr int kUnroll = G::kStream ? 1 : 8;
        // a contraction of operand X (modes or bond forces) into d
        auto with_x = [&](int res0, uint32_t d, bool first) {
#pragma unroll(kUnroll)
            for (int k = 0; k < G::KP / 16; ++k)
                block(res0 + k, d, x0 + (uint64_t)(k * (2 * 128 / 16)), G::XPART, id_x, first && k == 0);
        };
        const uint32_t d_u = tmem + e * G::ROWS, d_inc = d_u + NP * G::ROWS, d_z = G::kScaled ? d_inc + G::ROWS : d_inc;
        // a noise chunk: its turn of the buffer of its number mod 2
        auto with_z = [&](int sp, int ch) {
            const int b = ch & 1;
            wait(&n_ready[b], (sp * (G::NCH / 2) + (ch >> 1)) & 1, b != (int)rank);
            if constexpr (G::kPair) {
                // the other CTA's next chunk (no byte of it comes before both CTAs' MMAs have read this one)
                if (warp == 1 && leader && ok && b != (int)rank) mbar_expect_tx(&n_ready[b], z_bytes);
            }
#pragma unroll(G::kPair ? 1 : G::ZK / 16)
            for (int k = 0; k < G::ZK / 16; ++k)
                block(G::BLK + (G::ZK / 16) * ch + k, d_z, z0 + (uint64_t)(b * (G::ZB / 16) + k * (2 * G::ZLBO / 16)), G::ZPART,
                      id_z, ch == 0 && k == 0);
            if (leader && ok) {
                if constexpr (G::kPair) mma_commit_mc(&n_free[b], (uint16_t)(1u << b));     // to the CTA that draws this buffer
                else mma_commit(&n_free[b]);
            }
        };
        if constexpr (G::kPair) {
            if (warp == 1 && leader) mbar_expect_tx(&n_ready[rank ^ 1u], z_bytes);
        }
#pragma unroll 1
        for (int sp = 0; sp < a.n_steps && ok; ++sp) {
            wait(r_ready, sp & 1, false);
            with_x(0, d_u, true);
            if (leader && ok) mma_commit(u_done);
#pragma unroll 1
            for (int ch = 0; ch < (G::kPair ? 2 : G::NCH); ++ch) with_z(sp, ch);
            wait(v_ready, sp & 1, true);
            with_x(G::kScaled ? 0 : 2 * G::BLK, d_inc, G::kScaled);
            if constexpr (G::kPair) {
                // the later chunks, whose way between the CTAs passes behind the forward MMAs
#pragma unroll 1
                for (int ch = 2; ch < G::NCH; ++ch) with_z(sp, ch);
            }
            if (leader && ok) mma_commit(inc_done);
        }
    } else if (warp >= 2 && warp < 2 + kWork) {
        // ---------------- force and update
        const int q = warp & 3;                                 // TMEM lane quarter
        const int j = (32 * q + lane) & (M == 64 ? 63 : 127);   // bond (pair) and mode (pair) index
        // the tile's batches of four chains: this warp takes b0, b0 + bs, ... of its lanes
        const int b0 = ((warp - 2) >> 2) + (M == 64 ? 2 * (q >> 1) : 0), bs = M == 64 ? 4 : 2;
        const int nb = (Ct + 3) >> 2;
        const bool own0 = (32 * q & (M == 64 ? 63 : 127)) == 0 && lane == 0 && rank == 0;   // this thread holds mode 0
        // accumulator e's mode in this lane, and its K index in operand X past lane j's
        auto mode = [&](int e) { return G::kPair ? 2 * (128 * e + j) + (int)rank : NP * j + e; };
        auto xoff = [](int e) { return G::kPair ? e * 128 * 16 : e * 2 * G::XPART; };
        const uint32_t d_u = tmem + ((uint32_t)(32 * q) << 16), d_inc = d_u + NP * G::ROWS;
        auto col = [](int b) { return 24 * G::pair(b) + 4 * G::half(b); };     // the batch's first row
        uint8_t* xw = X + j * 16;
        const uint32_t xw_peer = G::kPair ? peer(xw) : 0u, u_peer = G::kPair ? peer(U) : 0u;
        const uint32_t v_peer = G::kPair ? peer(v_ready) : 0u, uin_peer = G::kPair ? peer(u_in) : 0u;
        float dm[NP], gw[NP], cs[NP], es[NP];
#pragma unroll
        for (int e = 0; e < NP; ++e) {
            const float4 c = la.lane_c[mode(e)];
            dm[e] = c.x; gw[e] = c.y; cs[e] = c.z; es[e] = c.w;
        }
        bool ok = true;
        auto arrive = [&](uint64_t* bar) {
            fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0 && ok) mbar_arrive(bar);
        };
        // the lanes agree on whether a wait was met, where TMEM loads, which are the whole
        // warp's, depend on it (those of the update run either way)
        auto agree = [&](bool met) { ok = __all_sync(0xffffffffu, met) != 0; };
        auto store_x = [&](uint2 hi, uint2 lo, int off, int ax, int b) {
            uint8_t* w = xw + off + (3 * G::pair(b) + ax) * G::XSBO + G::half(b) * 8;
            *reinterpret_cast<uint2*>(w) = hi;
            *reinterpret_cast<uint2*>(w + G::XPART) = lo;
        };
        // the modes (2 j, 2 j + 1) or j of a batch in global memory and in TMEM,
        // [parity][axis][chain]; chains past the tile's last are zero
        float* Rj = a.R + (size_t)3 * c0 * M + mode(0);
        auto load_r = [&](float (&r)[NP][3][4], int b) {
            const float* p = Rj + (size_t)(12 * b) * M;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool live = 4 * b + i < Ct;
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    if constexpr (G::kPair) {
                        r[0][ax][i] = live ? p[(3 * i + ax) * M] : 0.f;
                        r[NP - 1][ax][i] = live ? p[(3 * i + ax) * M + 256] : 0.f;
                    } else if constexpr (NP == 2) {
                        const float2 x = live ? *reinterpret_cast<const float2*>(p + (3 * i + ax) * M) : make_float2(0.f, 0.f);
                        r[0][ax][i] = x.x;
                        r[NP - 1][ax][i] = x.y;
                    } else {
                        r[0][ax][i] = live ? p[(3 * i + ax) * M] : 0.f;
                    }
                }
            }
        };
        auto store_r = [&](const float (&r)[NP][3][4], int b) {
            float* p = Rj + (size_t)(12 * b) * M;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (4 * b + i < Ct)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        if constexpr (G::kPair) {
                            p[(3 * i + ax) * M] = r[0][ax][i];
                            p[(3 * i + ax) * M + 256] = r[NP - 1][ax][i];
                        } else if constexpr (NP == 2)
                            *reinterpret_cast<float2*>(p + (3 * i + ax) * M) = make_float2(r[0][ax][i], r[NP - 1][ax][i]);
                        else
                            p[(3 * i + ax) * M] = r[0][ax][i];
                    }
        };
        const uint32_t r_col = d_u + G::kRCol;
        auto fetch_r = [&](float (&r)[NP][3][4], int b) {       // before a tmem_wait12
#pragma unroll
            for (int e = 0; e < NP; ++e)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) tmem_ld4(r_col + (b * NP + e) * 12 + 4 * ax, r[e][ax]);
        };
        auto keep_r = [&](const float (&r)[NP][3][4], int b) {
#pragma unroll
            for (int e = 0; e < NP; ++e)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) tmem_st4(r_col + (b * NP + e) * 12 + 4 * ax, r[e][ax]);
        };
        auto put_r = [&](const float (&r)[NP][3][4], int b) {
#pragma unroll
            for (int e = 0; e < NP; ++e)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    uint2 h, l;
                    if constexpr (G::kScaled) {
                        const float x[4] = {cs[e] * r[e][ax][0], cs[e] * r[e][ax][1], cs[e] * r[e][ax][2], cs[e] * r[e][ax][3]};
                        split4(x, h, l);
                    } else {
                        split4(r[e][ax], h, l);
                    }
                    store_x(h, l, xoff(e), ax, b);
                }
        };
        // bond vectors -> residual force v (Eq. e11) of a batch, two chains at a time
        // (packed FP32)
        // (a pair of CTAs: the other CTA's operand, [hi, lo][axis], into `there`)
        auto force4 = [&](int b, uint2 (&there)[2][3]) {
            float u[NP][3][4];                  // even and odd part
            if constexpr (G::kPair) {
                float own[3][4];
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_u + rank * G::ROWS + 8 * ax + col(b), own[ax]);
                tmem_wait12(own);
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    const float4 o = *reinterpret_cast<const float4*>(U + ((3 * b + ax) * 128 + j) * 16);
                    const float oth[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        u[0][ax][i] = rank ? oth[i] : own[ax][i];
                        u[NP - 1][ax][i] = rank ? own[ax][i] : oth[i];
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < NP; ++e)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_u + e * G::ROWS + 8 * ax + col(b), u[e][ax]);
#pragma unroll
                for (int e = 0; e < NP; ++e) tmem_wait12(u[e]);
            }
            uint2 xh[NP][3], xl[NP][3];
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                f32x2 w[NP][3];
#pragma unroll
                for (int e = 0; e < NP; ++e)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) w[e][ax] = pack2(u[e][ax][i], u[e][ax][i + 1]);
                if constexpr (NP == 2) {
                    f32x2 p[3], m[3];     // bonds j and M - j
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        p[ax] = add2(w[NP - 1][ax], w[0][ax]);
                        m[ax] = sub2(w[NP - 1][ax], w[0][ax]);
                    }
                    const f32x2 fp = add2(rsqrt2(fma2(p[0], p[0], fma2(p[1], p[1], mul2(p[2], p[2])))), both2(-a.c12nu));
                    const f32x2 fm = add2(rsqrt2(fma2(m[0], m[0], fma2(m[1], m[1], mul2(m[2], m[2])))), both2(-a.c12nu));
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        const f32x2 vm = mul2(m[ax], fm);
                        w[0][ax] = fma2(p[ax], fp, mul2(vm, both2(-1.0f)));      // even modes
                        w[NP - 1][ax] = fma2(p[ax], fp, vm);                     // odd modes
                    }
                } else {
                    const f32x2 f = add2(rsqrt2(fma2(w[0][0], w[0][0], fma2(w[0][1], w[0][1], mul2(w[0][2], w[0][2])))),
                                         both2(-a.c12nu));
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) w[0][ax] = j >= 1 ? mul2(w[0][ax], f) : 0ull;   // v_0 = 0
                }
#pragma unroll
                for (int e = 0; e < NP; ++e)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        if (i == 0) split2(w[e][ax], xh[e][ax].x, xl[e][ax].x);
                        else split2(w[e][ax], xh[e][ax].y, xl[e][ax].y);
                    }
            }
            if constexpr (G::kPair) {
                // K index 128 rank + j of both CTAs' operands: this CTA's parity here, the other there
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    store_x(rank ? xh[NP - 1][ax] : xh[0][ax], rank ? xl[NP - 1][ax] : xl[0][ax], (int)rank * 128 * 16, ax, b);
                    there[0][ax] = rank ? xh[0][ax] : xh[NP - 1][ax];
                    there[1][ax] = rank ? xl[0][ax] : xl[NP - 1][ax];
                }
            } else {
#pragma unroll
                for (int e = 0; e < NP; ++e)
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) store_x(xh[e][ax], xl[e][ax], xoff(e), ax, b);
            }
        };
        // pair: the bond vectors of the other CTA's lanes, to that CTA
        auto send4 = [&](int b) {
            float v[3][4];
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_u + (rank ^ 1u) * G::ROWS + 8 * ax + col(b), v[ax]);
            tmem_wait12(v);
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
                st_peer16(u_peer + ((3 * b + ax) * 128 + j) * 16,
                          make_uint4(__float_as_uint(v[ax][0]), __float_as_uint(v[ax][1]), __float_as_uint(v[ax][2]),
                                     __float_as_uint(v[ax][3])), uin_peer);
        };
        // update (Eqs. d3, btum) of a batch whose modes are in r (tm: in TMEM)
        auto update4 = [&](float (&r)[NP][3][4], int b, int sp, bool tm, bool plain) {
            float d[NP][3][4];
            if (tm) fetch_r(r, b);
#pragma unroll
            for (int e = 0; e < NP; ++e)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_inc + e * G::ROWS + 8 * ax + col(b), d[e][ax]);
            if constexpr (G::kScaled) {
                float dz[3][4];
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) tmem_ld4(d_inc + G::ROWS + 8 * ax + col(b), dz[ax]);
                tmem_wait12(d[0]);
                tmem_wait12(dz);
#pragma unroll
                for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                    for (int i = 0; i < 4; ++i) d[0][ax][i] = fmaf(es[0], d[0][ax][i], dz[ax][i]);
            } else {
#pragma unroll
                for (int e = 0; e < NP; ++e) tmem_wait12(d[e]);
            }
            if (tm) {
#pragma unroll
                for (int e = 0; e < NP; ++e) tmem_wait12(r[e]);
            }
            if (own0) {
#pragma unroll
                for (int ax = 0; ax < 3; ++ax)
                    *reinterpret_cast<float4*>(s_d0 + 32 * ax + 4 * b) = make_float4(d[0][ax][0], d[0][ax][1], d[0][ax][2], d[0][ax][3]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (plain || sp < s_left[4 * b + i]) {      // a chain at its stop step stays as it is
#pragma unroll
                    for (int e = 0; e < NP; ++e) {
                        const float ry = r[e][1][i];
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) r[e][ax][i] += fmaf(-dm[e], r[e][ax][i], d[e][ax][i]);
                        if (!plain) r[e][0][i] = fmaf(__fmul_rn(s_shf[4 * b + i], gw[e]), ry, r[e][0][i]);
                    }
                }
            }
            put_r(r, b);
            if (tm) keep_r(r, b);
            else if (ok) store_r(r, b);
        };

        // operand X of the first step
#pragma unroll 1
        for (int b = b0; b < nb; b += bs) {
            float r[NP][3][4];
            load_r(r, b);
            if (own0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) r[0][0][i] = r[0][1][i] = r[0][2][i] = 0.f;
            }
            put_r(r, b);
            if (b < G::TB) keep_r(r, b);
        }
        tmem_wait_st();
        arrive(r_ready);
#pragma unroll 1
        for (int sp = 0; sp < a.n_steps; ++sp) {
            agree(ok && mbar_wait(u_done, sp & 1, a.err, abort_flag));
            fence_after();
            if constexpr (G::kPair) {
#pragma unroll 1
                for (int b = b0; ok && b < nb; b += bs) send4(b);
                agree(ok && mbar_wait_cl(u_in, sp & 1, a.err, abort_flag));
            }
            uint2 there[2][3], held[2][3];
#pragma unroll 1
            for (int b = b0; ok && b < nb; b += bs) {
                force4(b, there);
                if constexpr (G::kPair) {
                    const uint32_t w = xw_peer + rank * (128 * 16) + 3 * G::pair(b) * G::XSBO;
                    if (b == b0 && b + bs < nb) {
                        // goes with the next batch
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) held[i][ax] = there[i][ax];
                    } else if (b == b0 + bs) {
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax)
                                st_peer16(w + ax * G::XSBO + i * G::XPART, make_uint4(held[i][ax].x, held[i][ax].y, there[i][ax].x, there[i][ax].y), v_peer);
                    } else {
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax)
                                st_peer8(w + ax * G::XSBO + i * G::XPART + G::half(b) * 8, there[i][ax], v_peer);
                    }
                }
            }
            arrive(v_ready);
            // a batch whose modes are in global memory is updated last; they come from L2
            // while the forward MMAs run
            float rg[NP][3][4];
            const int bg = b0 + bs * ((G::TB - b0 + bs - 1) / bs);      // this warp's first one
            if (G::TB < 8 && bg < nb) load_r(rg, bg);
            ok = ok && mbar_wait(inc_done, sp & 1, a.err, abort_flag);
            fence_after();
#pragma unroll 1
            for (int b = b0; b < min(nb, G::TB); b += bs) {
                float r[NP][3][4];
                if (steady) update4(r, b, sp, true, true);
                else update4(r, b, sp, true, false);
            }
            if constexpr (G::TB < 8) {
#pragma unroll 1
                for (int b = bg; b < nb; b += bs) {
                    if (b != bg) load_r(rg, b);
                    update4(rg, b, sp, false, steady);
                }
            }
            tmem_wait_st();
            arrive(r_ready);
        }
        // the state back to global memory; mode 0, whose table columns are zero, has only
        // summed up its noise (the centre of mass is warp 19's).  A non-finite mode stays
        // non-finite: looked at once per launch.
        bool finite = true;
#pragma unroll 1
        for (int b = b0; b < nb; b += bs) {
            float r[NP][3][4];
            if (b < G::TB) {
                fetch_r(r, b);
#pragma unroll
                for (int e = 0; e < NP; ++e) tmem_wait12(r[e]);
            } else {
                load_r(r, b);
            }
            if (own0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) r[0][0][i] = r[0][1][i] = r[0][2][i] = 0.f;
            }
            if (ok) store_r(r, b);
#pragma unroll
            for (int e = 0; e < NP; ++e)
#pragma unroll
                for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                    for (int i = 0; i < 4; ++i) finite = finite && (4 * b + i >= Ct || isfinite(r[e][ax][i]));
        }
        if (!finite) atomicOr(a.err, 1);
    } else if (warp >= 2 + kWork && warp < 2 + kWork + kNoise) {
        // ---------------- normals (Eq. b5), drawn ahead of the step, 32 K indices of
        // each parity at a time, into two buffers in turn.  A lane draws four
        // consecutive beads of a chain (three Philox calls) and, with the mirror
        // symmetry, their four mirror images, and writes the sums and differences as
        // 8 bytes of a row of the noise operand: 8 lanes fill a chain's row, a warp
        // takes four chains (a batch).
        const int nw = warp - 2 - kWork;
        const int t = lane & 7;
        bool ok = true;
        const uint32_t nr_peer = G::kPair ? peer(&n_ready[rank]) : 0u;
        // a pair's CTAs draw the chunks of a step in turn, each into its own buffer of
        // both CTAs (the sums for the even modes' CTA, the differences for the other)
        // (K = 32 at a time: half a chunk of a pair)
        constexpr int NDR = G::kPair ? G::KP / 64 : G::NCH;     // drawn by this CTA per step
        const int chunks = a.n_steps * NDR;
        static_assert(G::NCH % 2 == 0, "chunks in pairs");
        // Both chunks of a pair are drawn before either is written, so that the second
        // half of a step's normals waits in registers for the first half's MMAs.
#pragma unroll 1
        for (int chunk = 0; chunk < chunks; chunk += 2) {
            const int sp = chunk / NDR, ch = chunk - NDR * sp;
            uint2 hi[2][NP][3], lo[2][NP][3];
            // with fewer batches than warps, a chunk's batches go to other warps than the last one's
            const int cl[2] = {4 * ((nw + 5 * chunk) & (kNoise - 1)) + (lane >> 3),
                               4 * ((nw + 5 * chunk + 5) & (kNoise - 1)) + (lane >> 3)};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (cl[k] >= Ct) continue;
                const uint32_t job = s_job[cl[k]];
                const int64_t st = s_step[cl[k]] + sp;
                const uint32_t b4 = (uint32_t)(8 * (G::kPair ? 2 * ch + 2 * (int)rank + k : ch + k) + t);       // beads 4 b4 ...
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
                        split4(s, hi[k][0][ax], lo[k][0][ax]);
                        split4(d, hi[k][NP - 1][ax], lo[k][NP - 1][ax]);
                    }
                } else {
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) split4(z[ax], hi[k][0][ax], lo[k][0][ax]);
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                // the MMAs have read the chunk that this buffer held
                const int buf = G::kPair ? (int)rank : k;
                if constexpr (G::kPair) {
                    if (chunk > 0 && k == 0) ok = ok && mbar_wait_cl(&n_free[buf], ((chunk >> 1) - 1) & 1, a.err, abort_flag);
                } else {
                    if (chunk >= 2) ok = ok && mbar_wait(&n_free[buf], ((chunk >> 1) - 1) & 1, a.err, abort_flag);
                }
                if (cl[k] < Ct && ok) {
                    const int b = cl[k] >> 2;
                    uint8_t* w = Z + buf * G::ZB + ((G::kPair ? 4 * k : 0) + (t >> 1)) * G::ZLBO + 3 * G::pair(b) * 128 +
                                 (4 * G::half(b) + (cl[k] & 3)) * 16 + (t & 1) * 8;
                    if constexpr (G::kPair) {
                        const uint32_t wp = peer(w);
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) {
                            *reinterpret_cast<uint2*>(w + ax * 128) = rank ? hi[k][NP - 1][ax] : hi[k][0][ax];
                            *reinterpret_cast<uint2*>(w + G::ZPART + ax * 128) = rank ? lo[k][NP - 1][ax] : lo[k][0][ax];
                            st_peer8(wp + ax * 128, rank ? hi[k][0][ax] : hi[k][NP - 1][ax], nr_peer);
                            st_peer8(wp + G::ZPART + ax * 128, rank ? lo[k][0][ax] : lo[k][NP - 1][ax], nr_peer);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < NP; ++e)
#pragma unroll
                            for (int ax = 0; ax < 3; ++ax) {
                                *reinterpret_cast<uint2*>(w + e * 2 * G::ZPART + ax * 128) = hi[k][e][ax];
                                *reinterpret_cast<uint2*>(w + e * 2 * G::ZPART + G::ZPART + ax * 128) = lo[k][e][ax];
                            }
                    }
                }
                if (G::kPair && k == 0) continue;       // the two halves arrive together
                fence_proxy_async();
                __syncwarp();
                if (lane == 0 && ok) mbar_arrive(&n_ready[buf]);
            }
        }
        // a pair: the other CTA's last commits to this CTA's n_free have landed
        if constexpr (G::kPair) ok = ok && mbar_wait_cl(&n_free[rank], ((chunks >> 1) - 1) & 1, a.err, abort_flag);
    } else if (warp == 19) {
        // ---------------- the centre of mass (p = 0 of Eq. d3 with zeta_0 = 0) in
        // FP64, a chain per lane, and the step counters
        bool ok = true;
        const bool live = lane < Ct && rank == 0;       // a pair: the even modes' CTA
        double cm[3] = {0.0, 0.0, 0.0};
        double* cg = a.com + 3 * (size_t)(c0 + lane);
        if (live)
            for (int ax = 0; ax < 3; ++ax) cm[ax] = cg[ax];
        const double sh = __dmul_rn(s_shear[lane], a.dtau);
        // a pair: it also arms the barriers for the other CTA's stores of a step
        const uint32_t nb = (uint32_t)(Ct + 3) >> 2;
        auto arm = [&] {
            if constexpr (G::kPair) {
                mbar_expect_tx(u_in, nb * 128u * 48u);
                mbar_expect_tx(v_ready, nb * 128u * 48u);
            } else {
                mbar_arrive(v_ready);
            }
        };
        // every phase of r_ready in turn, and each before the arrival on v_ready that the
        // next one needs: armed first, the step could pass while this warp still looks for
        // phase 0, which then has the parity of phase 2
        ok = mbar_wait(r_ready, 0, a.err, abort_flag);
        if (lane == 0 && ok) arm();
#pragma unroll 1
        for (int sp = 0; sp < a.n_steps; ++sp) {
            ok = ok && mbar_wait(r_ready, (sp + 1) & 1, a.err, abort_flag);
            if (ok && live && sp < s_left[lane]) {
                const double ycm = cm[1];
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) cm[ax] = fma((double)s_d0[32 * ax + lane], a.inv_sqrtM, cm[ax]);
                if (has_shear) cm[0] = fma(sh, ycm, cm[0]);
            }
            __syncwarp();
            if (lane == 0 && ok && sp + 1 < a.n_steps) arm();
        }
        if (ok && live) {
            for (int ax = 0; ax < 3; ++ax) cg[ax] = cm[ax];
            a.step[c0 + lane] = s_step[lane] + s_left[lane];
        }
    }
    fence_before();
    __syncwarp();
    if constexpr (G::kPair) {
        // neither CTA leaves while the other may still write into its shared memory; after
        // a timeout, what this CTA has under way there lands first
        if (*abort_flag) {
            const uint64_t t0 = globaltimer();
            while (globaltimer() - t0 < 1000000ull) __nanosleep(1000);
        }
        __syncwarp();
        cluster_sync();
    } else {
        __syncthreads();
    }
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
