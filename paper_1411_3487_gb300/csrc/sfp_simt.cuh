// sfp_simt.cuh -- CUDA-core kernels of the mode-space step (FP32 and FP64).
//
// Layout of every per-chain array: [chain][axis][index], index contiguous,
// rows of length M (beads n or modes p).  A "row" j = 3*chain + axis.
#pragma once
#include "sfp_device.cuh"
#include "sfp_ptx.cuh"

namespace sfp {

// ---------------------------------------------------------------------------
// FP64 transform GEMM (NT):  Out[j][i] = sum_k In[j][k] * B[i][k]
//   inverse (Eq. e5):  In = R (k = p), B = chi  stored [n][p]  -> Out = u (bonds)
//   forward (Eq. c4):  In = f|z (k = n), B = phi^T stored [p][n] -> Out = DeltaH|Z
// Block tile BM rows x BN cols, K chunk BK; each thread owns TM x TN outputs.
// Any J, Ncols, K (ragged tails are zero-filled).
// ---------------------------------------------------------------------------
template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
k_gemm_nt(const double* __restrict__ In, const double* __restrict__ B, double* __restrict__ Out,
          int J, int Ncols, int K)
{
    constexpr int NT = (BM / TM) * (BN / TN);
    __shared__ double As[BK][BM + 1];
    __shared__ double Bs[BK][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid % (BN / TN), ty = tid / (BN / TN);
    const int j0 = blockIdx.y * BM, i0 = blockIdx.x * BN;
    double acc[TM][TN];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) acc[a][b] = 0.0;

    for (int k0 = 0; k0 < K; k0 += BK) {
        for (int e = tid; e < BM * BK; e += NT) {
            const int row = e / BK, kk = e % BK;
            const int gj = j0 + row, gk = k0 + kk;
            As[kk][row] = (gj < J && gk < K) ? In[(size_t)gj * K + gk] : 0.0;
        }
        for (int e = tid; e < BN * BK; e += NT) {
            const int row = e / BK, kk = e % BK;
            const int gi = i0 + row, gk = k0 + kk;
            Bs[kk][row] = (gi < Ncols && gk < K) ? B[(size_t)gi * K + gk] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[TM], b[TN];
#pragma unroll
            for (int x = 0; x < TM; ++x) a[x] = As[kk][ty * TM + x];
#pragma unroll
            for (int y = 0; y < TN; ++y) b[y] = Bs[kk][tx * TN + y];
#pragma unroll
            for (int x = 0; x < TM; ++x)
#pragma unroll
                for (int y = 0; y < TN; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < TM; ++x) {
        const int gj = j0 + ty * TM + x;
        if (gj >= J) continue;
#pragma unroll
        for (int y = 0; y < TN; ++y) {
            const int gi = i0 + tx * TN + y;
            if (gi < Ncols) Out[(size_t)gj * Ncols + gi] = acc[x][y];
        }
    }
}

// ---------------------------------------------------------------------------
// The FP64 transforms between beads and modes of chains with an even number of beads,
// in halves: phi_{n,p} is even (p even) or odd (p odd) under n -> M - 1 - n, so
//   DIR 0 (B = phi^T [p][n]):  R_p = sum_{n < M/2} phi_{n,p} (r_n +- r_{M-1-n})
//   DIR 1 (B = phi [n][p]):    r_n, r_{M-1-n} = E_n +- O_n, E and O the sums over the
//                              even and the odd modes, n < M/2
// take half the products of k_gemm_nt, which GB300's FP64 units bound: 4096 x 256
// beads 1557 us there, 804 us here.  Block tile 64 rows x 32 outputs of each parity.
// ---------------------------------------------------------------------------
template <int DIR>
__global__ void __launch_bounds__(256)
k_sym_gemm(const double* __restrict__ In, const double* __restrict__ B, double* __restrict__ Out, int J, int M)
{
    constexpr int BM = 64, BN = 32, BK = 8;
    __shared__ double As[2][BK][BM + 1];            // [parity]
    __shared__ double Bs[2][BK][BN + 1];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16, H = M / 2;
    const int j0 = blockIdx.y * BM, i0 = blockIdx.x * BN;
    double acc[2][4][2] = {};
    for (int k0 = 0; k0 < H; k0 += BK) {
        for (int e = tid; e < BM * BK; e += 256) {
            const int row = e / BK, kk = e % BK, j = j0 + row, k = k0 + kk;
            double x = 0.0, y = 0.0;
            if (j < J && k < H) {
                const double* p = In + (size_t)j * M;
                if constexpr (DIR == 0) {
                    const double u = p[k], v = p[M - 1 - k];
                    x = u + v;
                    y = u - v;
                } else {
                    x = p[2 * k];
                    y = p[2 * k + 1];
                }
            }
            As[0][kk][row] = x;
            As[1][kk][row] = y;
        }
        for (int e = tid; e < 2 * BN * BK; e += 256) {
            const int par = e / (BN * BK), col = (e / BK) % BN, kk = e % BK, i = i0 + col, k = k0 + kk;
            double x = 0.0;
            if (i < H && k < H) x = DIR == 0 ? B[(size_t)(2 * i + par) * M + k] : B[(size_t)i * M + 2 * k + par];
            Bs[par][kk][col] = x;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk)
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                double a[4], b[2];
#pragma unroll
                for (int x = 0; x < 4; ++x) a[x] = As[par][kk][ty + 16 * x];
#pragma unroll
                for (int y = 0; y < 2; ++y) b[y] = Bs[par][kk][tx + 16 * y];
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int y = 0; y < 2; ++y) acc[par][x][y] = fma(a[x], b[y], acc[par][x][y]);
            }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int j = j0 + ty + 16 * x;
        if (j >= J) continue;
        double* o = Out + (size_t)j * M;
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int i = i0 + tx + 16 * y;
            if (i >= H) continue;
            const double e = acc[0][x][y], d = acc[1][x][y];
            if constexpr (DIR == 0) {
                o[2 * i] = e;
                o[2 * i + 1] = d;
            } else {
                o[i] = e + d;
                o[M - 1 - i] = e - d;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The same product in FP32 (the plain path, and every length that the tensor-core
// kernels do not take): Out_z[j][i] = sum_k In_z[j][k] B_z[i][k], blockIdx.z picks the
// product (the forward transform's two are one launch).  Block tile BM x BN, K chunks
// of 16 in two shared-memory buffers (the next chunk's loads are in registers while
// one is multiplied), TM x TN outputs per thread as TM / 2 pairs of rows
// (fma.rn.f32x2); every output sums k in ascending order.  VEC: K % 4 == 0 and
// 16-byte-aligned operands (float4 loads and stores).
// Bound by FP32 issue on large shapes (48 of 80 TFLOP/s at 49152 x 512 x 512, 36 at
// 12288 x 256 x 256), by the latency of one block per SM on small ones (19 us for
// 3072 x 256 x 256, inverse).  With k_gemm_nt's 128 x 128 tiles (scalar loads, one
// buffer, 48 blocks on 152 SMs) a step of 1024 x 256 beads took 287 us, here 57; 2001
// x 100 beads 83 and 37, 4096 x 256 beads 396 and 142, 50 x 1000 beads 1099 and 107.
// ---------------------------------------------------------------------------
struct GemmF32 {
    const float* in[2];
    const float* b[2];
    float* out[2];
};

template <int BM, int BN, int TM, int TN, bool VEC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
k_gemm_f32(const GemmF32 g, int J, int N, int K)
{
    constexpr int NT = (BM / TM) * (BN / TN), BK = 16;
    constexpr int LA = BM + 4, LB = BN + 4;                     // row pitches of the k-major tiles
    constexpr int QA = BM * BK / 4 / NT, QB = BN * BK / 4 / NT; // float4 loads per thread and chunk
    static_assert(QA * NT * 4 == BM * BK && QB * NT * 4 == BN * BK && TM % 4 == 0 && TN % 4 == 0, "tile split");
    __shared__ __align__(16) float As[2][BK][LA];
    __shared__ __align__(16) float Bs[2][BK][LB];
    const float* __restrict__ In = blockIdx.z ? g.in[1] : g.in[0];
    const float* __restrict__ B = blockIdx.z ? g.b[1] : g.b[0];
    float* __restrict__ Out = blockIdx.z ? g.out[1] : g.out[0];
    const int tid = threadIdx.x, tx = tid % (BN / TN), ty = tid / (BN / TN);
    const int j0 = blockIdx.y * BM, i0 = blockIdx.x * BN;
    float4 ra[QA], rb[QB];
    auto fetch4 = [&](const float* __restrict__ p, int row, int rows, int k) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < rows) {
            const float* q = p + (size_t)row * K + k;
            if constexpr (VEC) {
                if (k < K) x = *reinterpret_cast<const float4*>(q);
            } else {
                if (k < K) x.x = q[0];
                if (k + 1 < K) x.y = q[1];
                if (k + 2 < K) x.z = q[2];
                if (k + 3 < K) x.w = q[3];
            }
        }
        return x;
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int e = tid + NT * q;
            ra[q] = fetch4(In, j0 + (e >> 2), J, k0 + 4 * (e & 3));
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = tid + NT * q;
            rb[q] = fetch4(B, i0 + (e >> 2), N, k0 + 4 * (e & 3));
        }
    };
    auto put = [&](int buf) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int e = tid + NT * q, m = e >> 2, k = 4 * (e & 3);
            As[buf][k][m] = ra[q].x; As[buf][k + 1][m] = ra[q].y; As[buf][k + 2][m] = ra[q].z; As[buf][k + 3][m] = ra[q].w;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = tid + NT * q, m = e >> 2, k = 4 * (e & 3);
            Bs[buf][k][m] = rb[q].x; Bs[buf][k + 1][m] = rb[q].y; Bs[buf][k + 2][m] = rb[q].z; Bs[buf][k + 3][m] = rb[q].w;
        }
    };
    f32x2 acc[TM / 2][TN];
#pragma unroll
    for (int x = 0; x < TM / 2; ++x)
#pragma unroll
        for (int y = 0; y < TN; ++y) acc[x][y] = 0ull;
    fetch(0);
    put(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += BK) {
        const bool more = k0 + BK < K;
        if (more) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            f32x2 a[TM / 2], b[TN];
#pragma unroll
            for (int x = 0; x < TM / 4; ++x) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&As[buf][kk][ty * TM + 4 * x]);
                a[2 * x] = v.x;
                a[2 * x + 1] = v.y;
            }
#pragma unroll
            for (int y = 0; y < TN / 4; ++y) {
                const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * TN + 4 * y]);
                b[4 * y] = both2(v.x); b[4 * y + 1] = both2(v.y); b[4 * y + 2] = both2(v.z); b[4 * y + 3] = both2(v.w);
            }
#pragma unroll
            for (int x = 0; x < TM / 2; ++x)
#pragma unroll
                for (int y = 0; y < TN; ++y) acc[x][y] = fma2(a[x], b[y], acc[x][y]);
        }
        if (more) {
            put(buf ^ 1);           // the other buffer's readers passed the last barrier
            __syncthreads();
            buf ^= 1;
        }
    }
#pragma unroll
    for (int x = 0; x < TM; ++x) {
        const int gj = j0 + ty * TM + x;
        if (gj >= J) continue;
        float o[TN];
#pragma unroll
        for (int y = 0; y < TN; ++y) {
            float lo, hi;
            unpack2(acc[x / 2][y], lo, hi);
            o[y] = x & 1 ? hi : lo;
        }
#pragma unroll
        for (int y = 0; y < TN; y += 4) {
            const int gi = i0 + tx * TN + y;
            float* q = Out + (size_t)gj * N + gi;
            if (VEC && N % 4 == 0) {
                if (gi < N) *reinterpret_cast<float4*>(q) = make_float4(o[y], o[y + 1], o[y + 2], o[y + 3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (gi + i < N) q[i] = o[y + i];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Residual bond force (Eqs. e4, e5, e11), from bond vectors:
//   u_n = sum_p chi_{n,p} R_p (given, n >= 1; slot 0 holds 0),
//   v_n = u_n (1/|u_n| - (1 - 2nu)) for n >= 1, v_0 = 0,
// so that DeltaH_p = sum_n chi_{n,p} v_n (Eq. e11) is the forward transform of
// v with the table chi^T.  The bond form needs no neighbour: each bond's force
// is its own, and the kernel is a stream of 12 B read and 12 B written per
// bond.  One thread per chain and quad of bonds 4t .. 4t+3; threads of a warp
// take consecutive quads, so each axis row moves as one coalesced run of
// float4 (VEC: M % 4 == 0).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void residual_v(const T u[3], bool ok, T c12nu, T v[3])
{
    const T l2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T s = ok ? rsqrt_t<T>(l2) - c12nu : T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] = u[a] * s;
}

template <typename T, bool VEC>
__device__ __forceinline__ void force_quad(const T* __restrict__ ub, T* __restrict__ vb, int C, int M, T c12nu, int64_t t)
{
    const int Q = (M + 3) >> 2;                    // bond quads per chain
    if (t >= (int64_t)C * Q) return;
    const int c = (int)(t / Q), n0 = 4 * (int)(t - (int64_t)c * Q);
    const size_t base = (size_t)c * 3 * M;
    T u[3][4];
    if constexpr (VEC) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float4 x = *reinterpret_cast<const float4*>(ub + base + (size_t)a * M + n0);
            u[a][0] = x.x; u[a][1] = x.y; u[a][2] = x.z; u[a][3] = x.w;
        }
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < 4; ++i) u[a][i] = n0 + i < M ? ub[base + (size_t)a * M + n0 + i] : T(0);
    }
    T v[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const T ui[3] = {u[0][i], u[1][i], u[2][i]};
        T vi[3];
        residual_v<T>(ui, n0 + i >= 1 && n0 + i < M, c12nu, vi);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a][i] = vi[a];
    }
    if constexpr (VEC) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            *reinterpret_cast<float4*>(vb + base + (size_t)a * M + n0) = make_float4(v[a][0], v[a][1], v[a][2], v[a][3]);
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (n0 + i < M) vb[base + (size_t)a * M + n0 + i] = v[a][i];
    }
}

// ---------------------------------------------------------------------------
// Bead noise (Eq. b5): z = the bead normals of (seed, job, step, tag 0); normal
// k = 3 n + alpha of a chain and step is value k % 4 of Philox call k / 4.
// With tag 2 the same kernel draws the mode-keyed noise Z (normal 3 p + alpha)
// straight into the mode-space noise buffer.
// One thread per chain and Philox call: its four normals land on two or three
// neighbouring beads, so the threads of a warp write ~43 consecutive beads of
// each axis row.  Bound by the Philox / Box-Muller arithmetic, not by its
// 12 B per bead; it does not depend on the state, so the staged step runs it
// beside the inverse transform.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void noise_call(T* __restrict__ z, int C, int M, uint32_t seed, const uint32_t* __restrict__ job,
                                           const int64_t* __restrict__ step, uint32_t tag, int64_t t)
{
    const int K = (3 * M + 3) >> 2;                // Philox calls per chain and step
    if (t >= (int64_t)C * K) return;
    const int c = (int)(t / K), call = (int)(t - (int64_t)c * K);
    T g[4];
    Normals<T>::draw4(seed, job[c], step[c], (uint32_t)call, tag, g);
    T* zc = z + (size_t)c * 3 * M;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = 4 * call + e, n = k / 3;
        if (n < M) zc[(size_t)(k - 3 * n) * M + n] = g[e];
    }
}

// The two as kernels of their own (the tensor-core transforms, whose inverse leaves
// the CUDA cores to the noise), and in one launch, the first nf blocks the force, the
// others the noise (the CUDA-core transforms, beside which noise on a second stream
// gains nothing: a step of 50 x 20 beads takes 20.9 us with the second stream's two
// event waits and 16.7 here, one of 1024 x 256 beads 59.3 and 57.0).
template <typename T, bool VEC>
__global__ void __launch_bounds__(256)
k_force(const T* __restrict__ ub, T* __restrict__ vb, int C, int M, T c12nu)
{
    force_quad<T, VEC>(ub, vb, C, M, c12nu, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T>
__global__ void __launch_bounds__(256)
k_noise(T* __restrict__ z, int C, int M, uint32_t seed, const uint32_t* __restrict__ job,
        const int64_t* __restrict__ step, uint32_t tag)
{
    noise_call<T>(z, C, M, seed, job, step, tag, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(256)
k_force_noise(const T* __restrict__ ub, T* __restrict__ vb, int C, int M, T c12nu, unsigned nf, T* __restrict__ z,
              uint32_t seed, const uint32_t* __restrict__ job, const int64_t* __restrict__ step, uint32_t tag)
{
    if (blockIdx.x < nf) force_quad<T, VEC>(ub, vb, C, M, c12nu, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    else noise_call<T>(z, C, M, seed, job, step, tag, (int64_t)(blockIdx.x - nf) * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
// Mode update (Eqs. d3, d6, f2, btum), one thread per (chain, mode), all axes:
//   p >= 1:  R += -dm_p R + h_p DeltaH_p + w_p Z_p ;  R^x += shear g_p R^y(old)
//   p == 0:  r_cm (FP64) += w_0 Z_0 / sqrt(M) ; x_cm += shear dtau y_cm(old);
//            the chain's step counter advances.
// dm_p = 1 - e^{-zeta_p dtau}; written as an increment so FP32 keeps the
// slow modes whose decay factor rounds to 1.
// ---------------------------------------------------------------------------
// V consecutive modes per thread (V = 4: float4 loads and stores, needs
// M % 4 == 0), chains along grid y (grid-stride).  With stop != NULL a chain
// advances only while step < stop, and the step counters are advanced
// afterwards by k_advance_steps (so that no thread of this kernel reads a
// counter that another one changes).
template <typename T, int V>
__device__ __forceinline__ void load_v(const T* p, T (&x)[V])
{
    if constexpr (V == 4 && sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) x[i] = p[i];
    }
}
template <typename T, int V>
__device__ __forceinline__ void store_v(T* p, const T (&x)[V])
{
    if constexpr (V == 4 && sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) p[i] = x[i];
    }
}

template <typename T, int V>
__global__ void __launch_bounds__(128)
k_mode_update(T* __restrict__ R, const T* __restrict__ DH, const T* __restrict__ ZM,
              double* __restrict__ com, int64_t* __restrict__ step,
              const T* __restrict__ dm, const T* __restrict__ h, const T* __restrict__ w,
              const T* __restrict__ g, const double* __restrict__ shear,
              int C, int M, double w0_cm, double dtau, int* __restrict__ bad,
              const int64_t* __restrict__ stop)
{
    const int p0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (p0 >= M) return;
    for (int c = blockIdx.y * blockDim.y + threadIdx.y; c < C; c += gridDim.y * blockDim.y) {
        // every load of the chain first (one memory round trip), the stop test after
        const size_t b = (size_t)c * 3 * M + p0;
        T r[3][V], y[3][V], zz[3][V], d[V], hh[V], ww[V], gg[V];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            load_v<T, V>(R + b + (size_t)a * M, r[a]);
            load_v<T, V>(DH + b + (size_t)a * M, y[a]);
            load_v<T, V>(ZM + b + (size_t)a * M, zz[a]);
        }
        load_v<T, V>(dm + p0, d);
        load_v<T, V>(h + p0, hh);
        load_v<T, V>(w + p0, ww);
        load_v<T, V>(g + p0, gg);
        const double sh = shear[c];
        const bool run = !stop || step[c] < stop[c];
        double cm[3] = {0.0, 0.0, 0.0};
        if (p0 == 0) {
#pragma unroll
            for (int a = 0; a < 3; ++a) cm[a] = com[3 * c + a];
        }
        if (!run) continue;
        // the FP64 shear rate is converted only for sheared chains (an integer test
        // of its bits: +0 and -0 mean no shear)
        const bool sheared = (__double_as_longlong(sh) << 1) != 0;
        T o[3][V];
        bool fin = true;
#pragma unroll
        for (int i = 0; i < V; ++i) {
#pragma unroll
            for (int a = 0; a < 3; ++a) o[a][i] = r[a][i] + fma(-d[i], r[a][i], fma(hh[i], y[a][i], ww[i] * zz[a][i]));
#pragma unroll
            for (int a = 0; a < 3; ++a) fin = fin && isfinite(o[a][i]);
        }
        if (sheared) {
            const T shT = (T)sh;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                o[0][i] += shT * gg[i] * r[1][i];
                fin = fin && isfinite(o[0][i]);
            }
        }
        if (p0 == 0) {
            // p = 0: the centre of mass in FP64 (zeta_0 = 0, Eq. d6 limit w_0;
            // w0_cm = w_0 / sqrt(M))
            com[3 * c] = cm[0] + w0_cm * (double)zz[0][0] + sh * dtau * cm[1];
            com[3 * c + 1] = cm[1] + w0_cm * (double)zz[1][0];
            com[3 * c + 2] = cm[2] + w0_cm * (double)zz[2][0];
#pragma unroll
            for (int a = 0; a < 3; ++a) o[a][0] = r[a][0];
            if (!stop) step[c] += 1;
        }
        if (!fin) atomicOr(bad, 1);
#pragma unroll
        for (int a = 0; a < 3; ++a) store_v<T, V>(R + b + (size_t)a * M, o[a]);
    }
}

// ---------------------------------------------------------------------------
// The whole mode-space step (Sec. 4) of one chain per CTA, n_steps per launch,
// on the CUDA cores (the FP64 path): the state stays in shared memory between
// steps, so a small batch (one chain) pays no launch per step.  Per step:
//   thread n (bead):  u_n = sum_p chi_{n,p} R_p (Eq. e5, all three axes from one
//                     pass over chiT[p][n]), v_n = u_n (1/|u_n| - (1 - 2nu)),
//                     v_0 = 0 (Eq. e11); threads c < 3M/4 draw Philox call c of
//                     the step (four bead normals, Eq. b5)
//   thread p (mode):  DeltaH_p = sum_n chi_{n,p} v_n, Z_p = sum_n phi_{n,p} z_n
//                     (Eqs. e11, c4), then R_p += -dm_p R_p + h_p DeltaH_p + w_p Z_p
//                     and the shear term g_p R^y_p on x (Eqs. d3, d6, f2, btum);
//                     p = 0 moves the FP64 centre of mass.
// Tables: chiT [p][n], chi [n][p], phi [n][p] (global, read through L1).  Shared
// memory: R, v, z as [3][M] each.  A chain advances only while step < stop.
// FOLD (M even): chi and phi are even or odd under n -> M - n and n -> M - 1 - n with
// the parity of p, so every sum runs over half the indices: thread 2 i + e sums the
// modes of parity e, its neighbour the others, and the two take bonds i and M - i (bond
// M / 2 its own image, in the place of bond 0); the forces come back as v_i -+ v_{M-i},
// the normals as z_n +- z_{M-1-n}.  FP64 issue bounds the kernel (about 60 cycles a warp
// instruction on a sub-partition): 512 chains of 128 beads 164 us a step without, 96
// with; 200 of 256 beads 308 and 167.
// ---------------------------------------------------------------------------
template <typename T, bool FOLD>
__global__ void __launch_bounds__(256)
k_chain_steps(T* __restrict__ Rg, double* __restrict__ com, int64_t* __restrict__ step,
              const int64_t* __restrict__ stop, const uint32_t* __restrict__ job,
              const double* __restrict__ shear, const T* __restrict__ chiT, const T* __restrict__ chi,
              const T* __restrict__ phi, const T* __restrict__ dm, const T* __restrict__ h,
              const T* __restrict__ w, const T* __restrict__ g, int C, int M, T c12nu, double w0_cm,
              double dtau, uint32_t seed, int n_steps, int mode_noise, int* __restrict__ bad)
{
    extern __shared__ unsigned char chain_smem[];
    T* sR = reinterpret_cast<T*>(chain_smem);     // [3][M]
    T* sv = sR + 3 * M;                           // [3][M]
    T* sz = sv + 3 * M;                           // [3][M]
    __shared__ double s_cm[3];
    const int c = blockIdx.x;
    if (c >= C) return;
    T* Rc = Rg + (size_t)c * 3 * M;
    for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) sR[i] = Rc[i];
    if (threadIdx.x < 3) s_cm[threadIdx.x] = com[3 * c + threadIdx.x];
    const uint32_t jb = job[c];
    const double sh = shear[c];
    const T shT = (T)sh;
    const int64_t st0 = step[c];
    const int64_t lim = stop ? stop[c] : INT64_MAX;
    const int n_calls = (3 * M + 3) >> 2;
    bool fin = true;
    __syncthreads();
    int s = 0;
    for (; s < n_steps && st0 + s < lim; ++s) {
        // bond vectors, bond forces, bead normals
        if constexpr (FOLD) {
            const int H = M / 2;
            for (int t0 = 0; t0 < M; t0 += blockDim.x) {
                const int t = min(t0 + (int)threadIdx.x, M - 1), i = t >> 1, e = t & 1, n = i ? i : H;
                T a0 = T(0), a1 = T(0), a2 = T(0);
                const T* __restrict__ x = chiT + (size_t)e * M + n;
                for (int p = e; p < M; p += 2, x += 2 * (size_t)M) {
                    const T c = *x;
                    a0 = fma(c, sR[p], a0);
                    a1 = fma(c, sR[M + p], a1);
                    a2 = fma(c, sR[2 * M + p], a2);
                }
                const T own[3] = {a0, a1, a2};
                T uu[3], vv[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const T oth = __shfl_xor_sync(0xffffffffu, own[a], 1);
                    uu[a] = e ? own[a] - oth : own[a] + oth;
                }
                residual_v<T>(uu, i > 0 || e == 0, c12nu, vv);      // bond 0 does not exist
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (i == 0 && e == 1) vv[a] = T(0);
                    const T oth = __shfl_xor_sync(0xffffffffu, vv[a], 1);
                    if (t0 + (int)threadIdx.x < M) sv[a * M + e * H + i] = e ? vv[a] + oth : vv[a] - oth;
                }
            }
        }
        for (int n = threadIdx.x; !FOLD && n < M; n += blockDim.x) {
            T u0 = T(0), u1 = T(0), u2 = T(0);
            for (int p = 1; p < M; ++p) {
                const T x = chiT[(size_t)p * M + n];
                u0 = fma(x, sR[p], u0);
                u1 = fma(x, sR[M + p], u1);
                u2 = fma(x, sR[2 * M + p], u2);
            }
            const T uu[3] = {u0, u1, u2};
            T vv[3];
            residual_v<T>(uu, n >= 1, c12nu, vv);
            sv[n] = vv[0]; sv[M + n] = vv[1]; sv[2 * M + n] = vv[2];
        }
        for (int k = threadIdx.x; k < n_calls; k += blockDim.x) {
            T gq[4];
            Normals<T>::draw4(seed, jb, st0 + s, (uint32_t)k, mode_noise ? 2u : 0u, gq);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int q = 4 * k + e;
                if (q < 3 * M) sz[(q % 3) * M + q / 3] = gq[e];
            }
        }
        __syncthreads();
        if (FOLD && !mode_noise) {
            // the normals as sums (first half) and differences (second half, mirrored)
            for (int k = threadIdx.x; k < 3 * (M / 2); k += blockDim.x) {
                const int a = k / (M / 2), n = k - a * (M / 2);
                const T x = sz[a * M + n], y = sz[a * M + M - 1 - n];
                sz[a * M + n] = x + y;
                sz[a * M + M - 1 - n] = x - y;
            }
            __syncthreads();
        }
        // forward transform and update, all three axes of mode p
        for (int p = threadIdx.x; p < M; p += blockDim.x) {
            T d0 = T(0), d1 = T(0), d2 = T(0), z0 = T(0), z1 = T(0), z2 = T(0);
            if constexpr (FOLD) {
                const int H = M / 2, e = p & 1;
                const T* v = sv + e * H;
                for (int k = 0; k < H; ++k) {
                    const T x = chi[(size_t)(k ? k : H) * M + p];
                    d0 = fma(x, v[k], d0);
                    d1 = fma(x, v[M + k], d1);
                    d2 = fma(x, v[2 * M + k], d2);
                    if (!mode_noise) {
                        const T f = phi[(size_t)k * M + p];
                        const int q = e ? M - 1 - k : k;
                        z0 = fma(f, sz[q], z0);
                        z1 = fma(f, sz[M + q], z1);
                        z2 = fma(f, sz[2 * M + q], z2);
                    }
                }
            }
            for (int n = 0; !FOLD && n < M; ++n) {
                const T x = chi[(size_t)n * M + p];
                d0 = fma(x, sv[n], d0);
                d1 = fma(x, sv[M + n], d1);
                d2 = fma(x, sv[2 * M + n], d2);
                if (!mode_noise) {
                    const T f = phi[(size_t)n * M + p];
                    z0 = fma(f, sz[n], z0);
                    z1 = fma(f, sz[M + n], z1);
                    z2 = fma(f, sz[2 * M + n], z2);
                }
            }
            if (mode_noise) {
                // mode-keyed noise: the drawn normals are Z itself
                z0 = sz[p];
                z1 = sz[M + p];
                z2 = sz[2 * M + p];
            }
            if (p == 0) {
                // centre of mass (zeta_0 = 0, Eq. d6 limit; w0_cm = w_0 / sqrt(M)), shear on x
                const double ycm = s_cm[1];
                s_cm[0] += w0_cm * (double)z0 + sh * dtau * ycm;
                s_cm[1] += w0_cm * (double)z1;
                s_cm[2] += w0_cm * (double)z2;
            } else {
                const T r0 = sR[p], r1 = sR[M + p], r2 = sR[2 * M + p];
                const T dd = dm[p], hh = h[p], ww = w[p];
                T o0 = r0 + fma(-dd, r0, fma(hh, d0, ww * z0));
                const T o1 = r1 + fma(-dd, r1, fma(hh, d1, ww * z1));
                const T o2 = r2 + fma(-dd, r2, fma(hh, d2, ww * z2));
                if (shT != T(0)) o0 += shT * g[p] * r1;
                fin = fin && isfinite(o0) && isfinite(o1) && isfinite(o2);
                sR[p] = o0; sR[M + p] = o1; sR[2 * M + p] = o2;
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) Rc[i] = (i % M == 0) ? T(0) : sR[i];
    if (threadIdx.x < 3) com[3 * c + threadIdx.x] = s_cm[threadIdx.x];
    if (threadIdx.x == 0) step[c] = st0 + s;
    if (!fin) atomicOr(bad, 1);
}

// ---------------------------------------------------------------------------
// The same FP64 step for a few chains, each on a cluster of G CTAs, so that a
// chain uses the FP64 units of G SMs: CTA r of a chain's cluster owns bonds
// and modes r S .. r S + S - 1 (S = ceil(M / G)) and keeps full copies of R
// and v in its shared memory; each owner writes its slice into every CTA of
// the cluster (distributed shared memory).  Per step:
//   owner r:  u_n, v_n of its bonds (Eqs. e5, e11) to every CTA; while they travel,
//             Z_p of its modes (Eq. c4) from the step's bead normals (Eq. b5), drawn
//             for all the steps of the launch beforehand by k_noise_steps;
//   owner r:  DeltaH_p of its modes (Eq. e11), the update of R_p (Eqs. d3, d6,
//             f2, btum; rank 0 the FP64 centre of mass), R_p to every CTA.
// A value is an asynchronous store that counts its bytes on the reader's mbarrier, so
// that a hand-over is one way through the cluster, without a fence or a barrier of all
// its threads.  A warp sends its part of one array only after all of the other has
// arrived, and every warp that reads an array sends a part of the other after its last
// read: neither array is overwritten while it is read, and no phase of a barrier begins
// before the one before it is over for everyone who waits on it.  That needs all of them
// to own something (M < G S leaves CTAs without bonds or modes, M <= 3 G warps): CTAs
// that own nothing take no part and are sent nothing, warps that own nothing do not wait.
// A CTA or warp that waits without being waited for can fall two phases behind, and the
// bytes of the second then keep the count of the first from ever being zero.
// What bounds it is latency, and most of that FP64 issue: a sub-partition of the SM takes
// about 60 cycles per FP64 warp instruction.  So a warp takes a bond or mode at a time, its
// lanes 8 a + j the sums of axis a, every eighth term each: one addition per step of the
// reduction instead of three, DeltaH_p and Z_p in one; the tables lie in shared memory,
// and the normals of the next step come in beside this one.
// The FP64 Box-Muller of a Philox call is a long dependent chain (~5 us), so the
// normals come from a separate kernel that draws every call of every step at once.
// One chain, us a step (cluster barriers, tables and normals from L2 before -> here): 64
// beads 6.6 -> 3.2, 128 11.8 -> 7.5, 256 29.4 -> 22.0; 8 chains of 64 beads 9.1 -> 4.5.
// Every wait is bounded; after a timeout the CTA raises bit 1 of the error word, its
// threads run through the remaining steps without sending or arming anything, and no CTA of the
// cluster writes anything back: the chain is as it was before the launch.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();       // .aligned: the whole warp at once
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p in the shared memory of CTA `rank` of the cluster (p: this CTA's own copy), counted on
// that CTA's mbarrier `bar`.
__device__ __forceinline__ void st_peer(const double* p, uint32_t rank, double v, uint64_t* bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                 ::"r"(ptx::mapa(ptx::smem_u32(p), rank)), "l"(__double_as_longlong(v)),
                 "r"(ptx::mapa(ptx::smem_u32(bar), rank)) : "memory");
}
__device__ __forceinline__ void copy_async8(double* dst, const double* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
// Sum over the lanes 8 a .. 8 a + 7 of an axis.
__device__ __forceinline__ double sum8(double x)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Shared memory of a CTA: R and v ([3][M + 8]: the axes in different banks), the normals
// of two steps, the tables of the owned bonds and modes and their dm, g, h, w.  Rows of
// the tables are a multiple of 8 long, and all rows zero from M on, so that the eight
// lanes of a sum take the same number of terms (with one more in some of them a warp runs
// the loop's two forms in turn: one chain of 63 beads 3.8 us a step as it is, 4.7 then).
__host__ __device__ constexpr int chain_cluster_pitch(int M) { return (M + 7) & ~7; }
constexpr size_t chain_cluster_bytes(int M, int G)
{
    const size_t S = (size_t)(M + G - 1) / G;
    return 8 * (12 * (size_t)(M + 8) + S * (3 * (size_t)chain_cluster_pitch(M) + 4));
}

template <int G>
__global__ void __launch_bounds__(128)
k_chain_cluster(double* __restrict__ Rg, double* __restrict__ com, int64_t* __restrict__ step,
                const int64_t* __restrict__ stop, const double* __restrict__ shear, const double* __restrict__ chiT,
                const double* __restrict__ chi, const double* __restrict__ phi, const double* __restrict__ dm,
                const double* __restrict__ h, const double* __restrict__ w, const double* __restrict__ g, int C,
                int M, double c12nu, double w0_cm, double dtau, int n_steps, const double* __restrict__ zpre,
                int mode_noise, int* __restrict__ bad, int stall_test)
{
    extern __shared__ unsigned char chain_smem[];
    const int P = M + 8, MP = chain_cluster_pitch(M);
    double* sR = reinterpret_cast<double*>(chain_smem);   // [3][P]
    double* sv = sR + 3 * P;                              // [3][P]
    double* sz = sv + 3 * P;                              // [2][3][P]
    double* tab = sz + 6 * P;                             // [S][3][MP] chi_n, chi_p, phi_p; [S] dm, g, h, w (w0_cm)
    __shared__ uint64_t v_in, r_in;                       // v, R of every CTA have arrived (1 + tx)
    __shared__ uint64_t never;                            // nothing arrives here (the stall test)
    __shared__ int s_abort;
    volatile int* abort_flag = &s_abort;
    const uint32_t rank = ptx::cluster_rank();
    const int c = blockIdx.x / G;                         // the cluster's chain (c < C: grid = G C)
    const int S = (M + G - 1) / G;
    const int lo = min(M, (int)rank * S), hi = min(M, lo + S), nown = hi - lo;
    const int nwarp = (int)blockDim.x / 32, wid = (int)threadIdx.x / 32, lane = (int)threadIdx.x % 32;
    const int j = lane & 7, ax = min(lane >> 3, 2);
    const bool sends = lane < 24;
    const int owners = (M + S - 1) / S;                   // CTAs 0 .. owners - 1 own something
    const bool owns = wid < nown;                         // this warp does (uniform; warp 0 of every owner)
    // every warp runs the same passes over the owned bonds / modes
    const int passes = (nown + nwarp - 1) / nwarp;
    double* tdm = tab + (size_t)S * 3 * MP;
    double *tg = tdm + S, *th = tg + S, *tw = th + S;
    double* Rc = Rg + (size_t)c * 3 * M;
    for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) sR[i / M * P + i % M] = Rc[i];
    // all copies under way at once (a call of one step of 12 chains of 256 beads: 74 us, 86
    // with loads through registers); phi by columns: a bead's owned modes lie side by side
    for (int o = wid; o < nown; o += nwarp)
        for (int k = lane; k < M; k += 32) {
            copy_async8(tab + (size_t)o * 3 * MP + k, chi + (size_t)(lo + o) * M + k);
            copy_async8(tab + (size_t)(o * 3 + 1) * MP + k, chiT + (size_t)(lo + o) * M + k);
        }
    for (int i = threadIdx.x, o = i % max(nown, 1), k = i / max(nown, 1); i < nown * M; i += blockDim.x) {
        copy_async8(tab + (size_t)(o * 3 + 2) * MP + k, phi + (size_t)k * M + lo + o);
        o += (int)blockDim.x;
        k += o / nown;
        o %= nown;
    }
    for (int i = threadIdx.x; i < 12 * 8; i += blockDim.x) sR[(i >> 3) * P + M + (i & 7)] = 0.0;     // R, v, normals
    for (int i = threadIdx.x; i < 3 * nown * 8; i += blockDim.x)
        if (M + (i & 7) < MP) tab[(size_t)(i >> 3) * MP + M + (i & 7)] = 0.0;
    for (int i = threadIdx.x; i < nown; i += blockDim.x) {
        tdm[i] = dm[lo + i];
        tg[i] = g[lo + i];
        th[i] = h[lo + i];
        tw[i] = lo + i ? w[lo + i] : w0_cm;
    }
    double cm = com[3 * c + ax];        // the centre of mass of this lane's axis (rank 0, warp 0)
    const double sh = shear[c];
    const int64_t st0 = step[c];
    const int64_t lim = stop ? stop[c] : INT64_MAX;
    bool fin = true, ok = true;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&v_in, 1);
        ptx::mbar_init(&r_in, 1);
        ptx::mbar_init(&never, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        ptx::mbar_expect_tx(&v_in, (uint32_t)(24 * M));
        ptx::mbar_expect_tx(&r_in, (uint32_t)(24 * (M - 1)));
    }
    auto fetch_z = [&](int s) {
        if (s < n_steps) {
            const double* src = zpre + ((size_t)s * C + c) * 3 * M;
            for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) copy_async8(sz + (s & 1) * 3 * P + i / M * P + i % M, src + i);
        }
    };
    fetch_z(0);
    asm volatile("cp.async.wait_all;" ::: "memory");
    // every CTA of the cluster runs (and has loaded R) before any remote write
    cluster_barrier();
    // stall test: the waits of one CTA run out here, and those of the others for its forces
    if (stall_test && (int)rank == owners - 1) ok = ptx::mbar_wait_cl(&never, 0, bad, abort_flag);
    int s = 0;
    for (; nown > 0 && s < n_steps && st0 + s < lim; ++s) {
        for (int pass = 0; pass < passes; ++pass) {
            const int gi = pass * nwarp + wid;
            if (gi >= nown) break;                      // the whole warp
            const int n = lo + gi;
            const double* t = tab + (size_t)gi * 3 * MP;
            double u = 0.0;
#pragma unroll 8
            for (int p = j; p < MP; p += 8) u = fma(t[p], sR[ax * P + p], u);       // chi_{n,0} = 0
            u = sum8(u);
            const double u0 = __shfl_sync(0xffffffffu, u, 0), u1 = __shfl_sync(0xffffffffu, u, 8),
                         u2 = __shfl_sync(0xffffffffu, u, 16);
            const double l2 = fma(u0, u0, fma(u1, u1, u2 * u2));
            const double v = n >= 1 ? u * (rsqrt_t<double>(l2) - c12nu) : 0.0;
            if (sends && ok)
#pragma unroll
                for (int r = j; r < G; r += 8)
                    if (r < owners) st_peer(&sv[ax * P + n], (uint32_t)r, v, &v_in);
        }
        const double* z = sz + (s & 1) * 3 * P;
        // this lane's part of w_p Z_p (w0_cm Z_0) of an owned mode
        auto noise = [&](int gi) {
            const int p = lo + gi;
            double x = 0.0;
            if (mode_noise) {
                if (j == 0) x = z[ax * P + p];
            } else {
                const double* t = tab + ((size_t)gi * 3 + 2) * MP;
#pragma unroll 8
                for (int n = j; n < MP; n += 8) x = fma(t[n], z[ax * P + n], x);
            }
            return tw[gi] * x;
        };
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();        // also: every warp is done with the normals of the last step
        fetch_z(s + 1);
        double x0 = owns ? noise(wid) : 0.0;
        if (owns) ok = ok && ptx::mbar_wait_cl(&v_in, s & 1, bad, abort_flag);
        if (threadIdx.x == 0 && ok) ptx::mbar_expect_tx(&v_in, (uint32_t)(24 * M));    // only a phase that is over
        __syncwarp();
        for (int pass = 0; pass < passes; ++pass) {
            const int gi = pass * nwarp + wid;
            if (gi >= nown) break;
            const int p = lo + gi;
            const double* t = tab + ((size_t)gi * 3 + 1) * MP;
            const double r = sR[ax * P + p], ry = sR[P + p];
            double d = 0.0;
            if (p > 0)                  // mode 0 takes no force, and nobody waits for its warp's read
#pragma unroll 8
                for (int n = j; n < MP; n += 8) d = fma(t[n], sv[ax * P + n], d);
            d = sum8(fma(th[gi], d, pass == 0 ? x0 : noise(gi)));
            if (p == 0) {
                // centre of mass (zeta_0 = 0, Eq. d6 limit; w0_cm = w_0 / sqrt(M)), shear on x
                const double ycm = __shfl_sync(0xffffffffu, cm, 8);
                cm += d;
                if (ax == 0) cm = fma(sh * dtau, ycm, cm);
            } else {
                double o = r + fma(-tdm[gi], r, d);
                if (sh != 0.0 && ax == 0) o = fma(sh * tg[gi], ry, o);
                fin = fin && isfinite(o);
                __syncwarp();       // every lane has read the mode before one of them sends the new one here
                if (sends && ok)
#pragma unroll
                    for (int q = j; q < G; q += 8)
                        if (q < owners) st_peer(&sR[ax * P + p], (uint32_t)q, o, &r_in);
            }
        }
        if (owns) ok = ok && ptx::mbar_wait_cl(&r_in, s & 1, bad, abort_flag);
        if (threadIdx.x == 0 && ok) ptx::mbar_expect_tx(&r_in, (uint32_t)(24 * (M - 1)));
        __syncwarp();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();        // the modes that the waiting warps have seen, for the others too
    if (*abort_flag) {
        // what is under way in the cluster lands first; the other CTAs learn of it
        const uint64_t t0 = ptx::globaltimer();
        while (ptx::globaltimer() - t0 < 1000000ull) __nanosleep(1000);
        if (threadIdx.x < G)
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(ptx::mapa(ptx::smem_u32(&s_abort), threadIdx.x)), "r"(1) : "memory");
    }
    // nobody leaves while another CTA may still write into its shared memory
    cluster_barrier();
    if (*abort_flag) return;
    // each CTA writes back its own modes; rank 0 the centre of mass and the counter
    for (int i = threadIdx.x; i < 3 * nown; i += blockDim.x) {
        const int a = i / nown, p = lo + i % nown;
        Rc[a * M + p] = p == 0 ? 0.0 : sR[a * P + p];
    }
    if (rank == 0 && wid == 0 && sends && j == 0) com[3 * c + ax] = cm;
    if (rank == 0 && threadIdx.x == 0) step[c] = st0 + s;
    if (!fin) atomicOr(bad, 1);
}

// The cluster step of chains whose tables no CTA's shared memory holds (more than 352
// beads on 16 CTAs), or whose clusters would not all fit on the GPU with them: bound by FP64 issue and by the tables from L2 rather than by
// latency.  Q threads share the sums of one bond or mode, all three axes (Q a power of 2
// within a warp; neighbouring groups read neighbouring table entries), and the groups are
// dealt round-robin over the four warps, so that all four sub-partitions have FP64 work;
// plain stores to the other CTAs and a cluster barrier after each array.  (512 beads: 99
// us a step; with the lanes and hand-overs of k_chain_cluster, tables from L2, 121.)
// *p in the shared memory of CTA `rank` of the cluster (p: this CTA's own copy).
__device__ __forceinline__ void st_peer_wait(const double* p, uint32_t rank, double v)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
}

template <int G>
__global__ void __launch_bounds__(128)
k_chain_cluster_wide(double* __restrict__ Rg, double* __restrict__ com, int64_t* __restrict__ step,
                const int64_t* __restrict__ stop, const double* __restrict__ shear, const double* __restrict__ chiT,
                const double* __restrict__ chi, const double* __restrict__ phi, const double* __restrict__ dm,
                const double* __restrict__ h, const double* __restrict__ w, const double* __restrict__ g, int C,
                int M, double c12nu, double w0_cm, double dtau, int n_steps, const double* __restrict__ zpre,
                int mode_noise, int* __restrict__ bad, int)
{
    extern __shared__ unsigned char chain_smem[];
    double* sR = reinterpret_cast<double*>(chain_smem);   // [3][M]
    double* sv = sR + 3 * M;                              // [3][M]
    double* sz = sv + 3 * M;                              // [3][M]
    __shared__ double s_cm[3];
    const uint32_t rank = ptx::cluster_rank();
    const int c = blockIdx.x / G;                         // the cluster's chain (c < C: grid = G C)
    const int S = (M + G - 1) / G;
    const int lo = min(M, (int)rank * S), hi = min(M, lo + S), nown = hi - lo;
    int Q = 1;
    while (Q < 32 && 2 * Q * max(nown, 1) <= (int)blockDim.x) Q *= 2;
    const int nwarp = (int)blockDim.x / 32, wid = (int)threadIdx.x / 32, lane = (int)threadIdx.x % 32;
    const int grp = (lane / Q) * nwarp + wid, j = lane % Q, nG = (int)blockDim.x / Q;
    // every thread runs the same passes over the owned bonds / modes (groups past
    // nown compute zeros), so the shuffles always see full warps
    const int passes = (nown + nG - 1) / nG;
    double* Rc = Rg + (size_t)c * 3 * M;
    for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) sR[i] = Rc[i];
    if (threadIdx.x < 3) s_cm[threadIdx.x] = com[3 * c + threadIdx.x];
    const double sh = shear[c];
    const int64_t st0 = step[c];
    const int64_t lim = stop ? stop[c] : INT64_MAX;
    bool fin = true;
    // every CTA of the cluster runs (and has loaded R) before any remote write
    cluster_barrier();
    int s = 0;
    for (; s < n_steps && st0 + s < lim; ++s) {
        const double* zs = zpre + ((size_t)s * C + c) * 3 * M;
        for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) sz[i] = zs[i];
        for (int pass = 0; pass < passes; ++pass) {
            const int gi = pass * nG + grp;
            const bool act = gi < nown;
            const int n = act ? lo + gi : 0;
            double u0 = 0.0, u1 = 0.0, u2 = 0.0;
            for (int p = 1 + j; act && p < M; p += Q) {
                const double x = chiT[(size_t)p * M + n];
                u0 = fma(x, sR[p], u0);
                u1 = fma(x, sR[M + p], u1);
                u2 = fma(x, sR[2 * M + p], u2);
            }
            for (int o = Q / 2; o > 0; o >>= 1) {
                u0 += __shfl_xor_sync(0xffffffffu, u0, o);
                u1 += __shfl_xor_sync(0xffffffffu, u1, o);
                u2 += __shfl_xor_sync(0xffffffffu, u2, o);
            }
            const double uu[3] = {u0, u1, u2};
            double vv[3];
            residual_v<double>(uu, n >= 1, c12nu, vv);
            for (int r = j; act && r < G; r += Q)
                for (int a = 0; a < 3; ++a) st_peer_wait(&sv[a * M + n], (uint32_t)r, vv[a]);
        }
        cluster_barrier();
        for (int pass = 0; pass < passes; ++pass) {
            const int gi = pass * nG + grp;
            const bool act = gi < nown;
            const int p = act ? lo + gi : 0;
            double d0 = 0.0, d1 = 0.0, d2 = 0.0, z0 = 0.0, z1 = 0.0, z2 = 0.0;
            for (int n = j; act && n < M; n += Q) {
                const double x = chi[(size_t)n * M + p];
                d0 = fma(x, sv[n], d0);
                d1 = fma(x, sv[M + n], d1);
                d2 = fma(x, sv[2 * M + n], d2);
                if (!mode_noise) {
                    const double f = phi[(size_t)n * M + p];
                    z0 = fma(f, sz[n], z0);
                    z1 = fma(f, sz[M + n], z1);
                    z2 = fma(f, sz[2 * M + n], z2);
                }
            }
            if (mode_noise && act && j == 0) {
                // mode-keyed noise: Z_p itself (taken once per group)
                z0 = sz[p];
                z1 = sz[M + p];
                z2 = sz[2 * M + p];
            }
            for (int o = Q / 2; o > 0; o >>= 1) {
                d0 += __shfl_xor_sync(0xffffffffu, d0, o);
                d1 += __shfl_xor_sync(0xffffffffu, d1, o);
                d2 += __shfl_xor_sync(0xffffffffu, d2, o);
                z0 += __shfl_xor_sync(0xffffffffu, z0, o);
                z1 += __shfl_xor_sync(0xffffffffu, z1, o);
                z2 += __shfl_xor_sync(0xffffffffu, z2, o);
            }
            if (!act) {
                // a group past the owned modes: nothing to update
            } else if (p == 0) {
                // centre of mass (zeta_0 = 0, Eq. d6 limit; w0_cm = w_0 / sqrt(M)), shear on x
                if (j == 0) {
                    const double ycm = s_cm[1];
                    s_cm[0] += w0_cm * z0 + sh * dtau * ycm;
                    s_cm[1] += w0_cm * z1;
                    s_cm[2] += w0_cm * z2;
                }
            } else {
                const double r0 = sR[p], r1 = sR[M + p], r2 = sR[2 * M + p];
                const double dd = dm[p], hh = h[p], ww = w[p];
                double o0 = r0 + fma(-dd, r0, fma(hh, d0, ww * z0));
                const double o1 = r1 + fma(-dd, r1, fma(hh, d1, ww * z1));
                const double o2 = r2 + fma(-dd, r2, fma(hh, d2, ww * z2));
                if (sh != 0.0) o0 += sh * g[p] * r1;
                fin = fin && isfinite(o0) && isfinite(o1) && isfinite(o2);
                for (int r = j; r < G; r += Q) {
                    st_peer_wait(&sR[p], (uint32_t)r, o0);
                    st_peer_wait(&sR[M + p], (uint32_t)r, o1);
                    st_peer_wait(&sR[2 * M + p], (uint32_t)r, o2);
                }
            }
        }
        cluster_barrier();
    }
    // each CTA writes back its own modes; rank 0 the centre of mass and the counter
    for (int i = threadIdx.x; i < 3 * nown; i += blockDim.x) {
        const int a = i / nown, p = lo + i % nown;
        Rc[a * M + p] = p == 0 ? 0.0 : sR[a * M + p];
    }
    if (rank == 0 && threadIdx.x < 3) com[3 * c + threadIdx.x] = s_cm[threadIdx.x];
    if (rank == 0 && threadIdx.x == 0) step[c] = st0 + s;
    if (!fin) atomicOr(bad, 1);
}

// Bead normals of n_steps consecutive steps for the FP64 cluster path (Eq. b5):
// z[s][c][3][M] = the normals of chain c at step step[c] + s, one thread per
// (step, chain, Philox call); tag 2: the mode-keyed noise Z instead.
__global__ void __launch_bounds__(256)
k_noise_steps(double* __restrict__ z, int C, int M, uint32_t seed, const uint32_t* __restrict__ job,
              const int64_t* __restrict__ step, int n_steps, uint32_t tag)
{
    const int K = (3 * M + 3) >> 2;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_steps * C * K) return;
    const int call = (int)(t % K);
    const int64_t sc = t / K;
    const int c = (int)(sc % C), s = (int)(sc / C);
    double gq[4];
    Normals<double>::draw4(seed, job[c], step[c] + s, (uint32_t)call, tag, gq);
    double* zc = z + ((size_t)s * C + c) * 3 * M;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = 4 * call + e, n = k / 3;
        if (n < M) zc[(size_t)(k - 3 * n) * M + n] = gq[e];
    }
}

// step[c] += 1 for chains still below their stop step (after k_mode_update).
__global__ void k_advance_steps(int64_t* __restrict__ step, const int64_t* __restrict__ stop, int C)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < C && step[c] < stop[c]) step[c] += 1;
}

// ---------------------------------------------------------------------------
// Equilibrium start, FP64 (Philox counter (0,0,k,1)):
//   l = l0 + sqrt(T*) L^-T eps   with (I - nu A) = L L^T  (Ld diag, Lo sub-diag)
//   t_1 uniform on the sphere, t_n ~ von Mises-Fisher(t_{n-1}, nu l_{n-1} l_n / T*)
//   r_n = sum_{k<=n} l_k t_k, centroid removed.
// A block samples n_ch chains in shared memory, eq_pitch(M) doubles per chain: bond
// lengths [M], then turns and later positions [M][3]; the centroid ends in the first
// three lengths' place.  Only what is a chain of dependences stays serial, one thread
// per chain: the back substitution and the frame that each bond passes on to the next;
// Philox, logarithms, exponentials and sines run a bead per thread.  Bound by FP64
// issue (about 450 FP64 instructions per bead at 4 GFMA/s per SM).  One thread per
// chain for everything, in strided global memory, took 2367 us for 4096 x 256 beads;
// 845 us here.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int eq_pitch(int M) { return 4 * M + 1; }   // odd: chains apart in the banks

__device__ __forceinline__ void sample_starts(double* eq_smem, const double* __restrict__ l0, const double* __restrict__ Ld,
                                              const double* __restrict__ Lo, int n_ch, int M, double Tstar, double nu,
                                              uint32_t seed, const uint32_t* __restrict__ job)
{
    const int N = M - 1, pitch = eq_pitch(M);
    const double sT = sqrt(Tstar);
    // eps_i, the normal of bond i + 1
    for (int t = threadIdx.x; t < n_ch * N; t += blockDim.x) {
        const int c = t / N, i = t - c * N;
        const uint4 wd = philox4x32_10(make_uint4(0u, 0u, (uint32_t)(i + 1), 1u), make_uint2(seed, job[c]));
        double s, co;
        sincospi(2.0 * u01d(wd.y), &s, &co);
        eq_smem[c * pitch + i] = sqrt(-2.0 * log(u01d(wd.x))) * co;
    }
    __syncthreads();
    // back substitution L^T x = eps, then the bond lengths l = l0 + sqrt(T*) x
    if (threadIdx.x < n_ch) {
        double* x = eq_smem + threadIdx.x * pitch;
        double nxt = 0.0;
        for (int i = N - 1; i >= 0; --i) {
            const double v = (x[i] - nxt) / Ld[i];
            x[i] = l0[i] + sT * v;
            nxt = Lo[i] * v;
        }
    }
    __syncthreads();
    // turn of bond n against bond n - 1 (von Mises-Fisher): cosine, and sine times the
    // cosine and sine of the angle about bond n - 1
    for (int t = threadIdx.x; t < n_ch * (N - 1); t += blockDim.x) {
        const int c = t / (N - 1), n = 2 + t - c * (N - 1);
        const double* l = eq_smem + c * pitch;
        double* a = eq_smem + c * pitch + M + 3 * n;
        double ct = 1.0, ca = 0.0, sa = 0.0;
        if (Tstar > 0.0) {
            const uint4 wd = philox4x32_10(make_uint4(0u, 0u, (uint32_t)n, 1u), make_uint2(seed, job[c]));
            const double kap = nu * l[n - 2] * l[n - 1] / Tstar;
            const double U = u01d(wd.z);
            ct = 1.0 + log(U + (1.0 - U) * exp(-2.0 * kap)) / kap;
            const double st = sqrt(fmax(0.0, (1.0 - ct) * (1.0 + ct)));
            double sp, cp;
            sincospi(2.0 * u01d(wd.w), &sp, &cp);
            ca = st * cp;
            sa = st * sp;
        }
        a[0] = ct; a[1] = ca; a[2] = sa;
    }
    __syncthreads();
    // bond by bond along the chain; position n takes the place of turn n
    if (threadIdx.x < n_ch) {
        const double* l = eq_smem + threadIdx.x * pitch;
        double* a = eq_smem + threadIdx.x * pitch + M;
        const uint4 wd = philox4x32_10(make_uint4(0u, 0u, 0u, 1u), make_uint2(seed, job[threadIdx.x]));
        const double z0 = 2.0 * u01d(wd.x) - 1.0;
        const double st = sqrt((1.0 - z0) * (1.0 + z0));
        double sp, cp;
        sincospi(2.0 * u01d(wd.y), &sp, &cp);
        double t[3] = {st * cp, st * sp, z0}, acc[3] = {0.0, 0.0, 0.0}, sum[3] = {0.0, 0.0, 0.0};
        a[0] = a[1] = a[2] = 0.0;
        for (int n = 1; n <= N; ++n) {
            if (n >= 2 && Tstar > 0.0) {
                // orthonormal pair perpendicular to t (Duff et al., JCGT 2017)
                const double ct = a[3 * n], ca = a[3 * n + 1], sa = a[3 * n + 2];
                const double sg = copysign(1.0, t[2]);
                const double q = -1.0 / (sg + t[2]);
                const double bb = t[0] * t[1] * q;
                const double tn[3] = {ct * t[0] + ca * (1.0 + sg * t[0] * t[0] * q) + sa * bb,
                                      ct * t[1] + ca * (sg * bb) + sa * (sg + t[1] * t[1] * q),
                                      ct * t[2] - ca * (sg * t[0]) - sa * t[1]};
                const double inv = rsqrt(tn[0] * tn[0] + tn[1] * tn[1] + tn[2] * tn[2]);
#pragma unroll
                for (int k = 0; k < 3; ++k) t[k] = tn[k] * inv;
            }
            const double ln = l[n - 1];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                acc[k] += ln * t[k];
                a[3 * n + k] = acc[k];
                sum[k] += acc[k];
            }
        }
        // the centroid in the place of the first bond lengths (N >= 2), read below
        double* m = eq_smem + threadIdx.x * pitch;
#pragma unroll
        for (int k = 0; k < 3; ++k) m[k] = sum[k] / M;
    }
    __syncthreads();
}

// Starts of a batch, `per` chains per block.   out: pos[c][3][M]
__global__ void __launch_bounds__(256)
k_equilibrium(double* __restrict__ pos, const double* __restrict__ l0, const double* __restrict__ Ld,
              const double* __restrict__ Lo, int C, int M, int per, double Tstar, double nu, uint32_t seed,
              const uint32_t* __restrict__ job)
{
    extern __shared__ double eq_smem[];
    const int c0 = blockIdx.x * per, n_ch = min(per, C - c0);
    sample_starts(eq_smem, l0, Ld, Lo, n_ch, M, Tstar, nu, seed, job + c0);
    for (int t = threadIdx.x; t < n_ch * 3 * M; t += blockDim.x) {
        const int c = t / (3 * M), e = t - c * 3 * M, k = e / M, n = e - k * M;
        const double* q = eq_smem + c * eq_pitch(M);
        pos[(size_t)(c0 + c) * 3 * M + e] = q[M + 3 * n + k] - q[k];
    }
}

// Serving: start n chains in the slots slot[i] with job key jobv[i], stop step
// stopv[i] and shear rate shv[i] (1/tau).  One block per slot: it draws the
// equilibrium start in shared memory (eq_pitch(M) doubles) and projects it
// onto the modes R_p = sum_n phi_{n,p} r_n (Eq. c1, p >= 1; phi FP64 [n][p]); the
// centre of mass is at the origin and the step counter 0.
template <typename T>
__global__ void k_init_slots(T* __restrict__ R, double* __restrict__ com, int64_t* __restrict__ step,
                             int64_t* __restrict__ stop, uint32_t* __restrict__ job, double* __restrict__ shear,
                             const int32_t* __restrict__ slot, const uint32_t* __restrict__ jobv,
                             const int64_t* __restrict__ stopv, const double* __restrict__ shv,
                             const double* __restrict__ phi, const double* __restrict__ l0,
                             const double* __restrict__ Ld, const double* __restrict__ Lo,
                             int M, double Tstar, double nu, uint32_t seed)
{
    extern __shared__ double sh_pos[];
    const int i = blockIdx.x;
    const int c = slot[i];
    sample_starts(sh_pos, l0, Ld, Lo, 1, M, Tstar, nu, seed, jobv + i);
    T* Rc = R + (size_t)c * 3 * M;
    for (int p = threadIdx.x; p < M; p += blockDim.x) {
        double s[3] = {0.0, 0.0, 0.0};
        if (p > 0)
            for (int n = 0; n < M; ++n) {
                const double f = phi[(size_t)n * M + p];
#pragma unroll
                for (int a = 0; a < 3; ++a) s[a] += f * (sh_pos[M + 3 * n + a] - sh_pos[a]);
            }
#pragma unroll
        for (int a = 0; a < 3; ++a) Rc[(size_t)a * M + p] = (T)s[a];
    }
    if (threadIdx.x == 0) {
        com[3 * c] = com[3 * c + 1] = com[3 * c + 2] = 0.0;
        step[c] = 0;
        stop[c] = stopv[i];
        job[c] = jobv[i];
        shear[c] = shv[i];
    }
}

// Serving: copy the state of slots slot[i] to out[i][3][M] (FP64, R_0 = sqrt(M) r_cm),
// their centres of mass to cm[i][3] and step counters to st[i].
template <typename T>
__global__ void k_gather_slots(const T* __restrict__ R, const double* __restrict__ com,
                               const int64_t* __restrict__ step, const int32_t* __restrict__ slot, int n, int M,
                               double* __restrict__ out, double* __restrict__ cm, int64_t* __restrict__ st)
{
    const int i = blockIdx.x;
    if (i >= n) return;
    const int c = slot[i];
    const double sq = sqrt((double)M);
    for (int e = threadIdx.x; e < 3 * M; e += blockDim.x) {
        const int a = e / M, p = e % M;
        out[(size_t)i * 3 * M + e] = (p == 0) ? com[3 * c + a] * sq : (double)R[(size_t)c * 3 * M + e];
    }
    if (threadIdx.x < 3) cm[3 * i + threadIdx.x] = com[3 * c + threadIdx.x];
    if (threadIdx.x == 0) st[i] = step[c];
}

// ---------------------------------------------------------------------------
// Small conversion kernels.
// ---------------------------------------------------------------------------
// modes (S = FP64 or FP32, packed rows incl. p = 0) -> state R (T, p = 0
// zeroed) + r_cm
template <typename S, typename T>
__global__ void k_load_modes(const S* __restrict__ src, T* __restrict__ R,
                             double* __restrict__ com, int C, int M, double inv_sqrtM)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)C * 3 * M) return;
    const int p = (int)(t % M);
    const int64_t row = t / M;
    if (p == 0) {
        com[row] = (double)src[t] * inv_sqrtM;
        R[t] = T(0);
    } else {
        R[t] = (T)src[t];
    }
}

// state -> modes (D = FP64 or FP32, R_0 = sqrt(M) r_cm), chain c at off[c] (NULL: 3 c M)
template <typename T, typename D>
__global__ void k_store_modes(const T* __restrict__ R, const double* __restrict__ com,
                              D* __restrict__ dst, const int64_t* __restrict__ off, int C, int M, double sqrtM)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)C * 3 * M) return;
    const int p = (int)(t % M);
    const int64_t o = off ? off[t / M / 3] + t % (3 * (int64_t)M) : t;
    dst[o] = (p == 0) ? (D)(com[t / M] * sqrtM) : (D)R[t];
}

template <typename T>
__global__ void k_to_double(const T* __restrict__ a, double* __restrict__ b, int64_t n)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) b[t] = (double)a[t];
}

// positions (FP64 scaled, CoM-relative) + CoM -> observables i-iii per chain
__global__ void k_shape(const double* __restrict__ pos, int C, int M, double* __restrict__ out,
                        double d2)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const int N = M - 1, mb = (N + 1) / 2, mm = N / 2;
    const double* p = pos + (size_t)c * 3 * M;
    double L2 = 0, u2 = 0, m2 = 0;
    for (int a = 0; a < 3; ++a) {
        const double L = p[a * M + N] - p[a * M];
        const double u = p[a * M + mb] - p[a * M + mb - 1];
        const double m = p[a * M + mm];
        L2 += L * L; u2 += u * u; m2 += m * m;
    }
    out[4 * c + 0] = L2 * d2; out[4 * c + 1] = u2 * d2; out[4 * c + 2] = m2 * d2;
}

__global__ void k_philox_words(uint32_t seed, uint32_t job, int64_t step, uint32_t tag, int n,
                               uint32_t* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 w = philox4x32_10(
        make_uint4((uint32_t)step, (uint32_t)((uint64_t)step >> 32), (uint32_t)i, tag), make_uint2(seed, job));
    out[4 * i] = w.x; out[4 * i + 1] = w.y; out[4 * i + 2] = w.z; out[4 * i + 3] = w.w;
}

}  // namespace sfp

namespace sfp {

// ---------------------------------------------------------------------------
// Observable sampling (Sec. 5B, observables i-iii), one warp per chain, read
// from the mode state only:
//   L     = r_N - r_0       = sum_p (phi_{N,p} - phi_{0,p}) R_p
//   u_m   (middle bond)     = sum_p chi_{m,p} R_p,          m = ceil(N/2)
//   r_m - r_cm (middle bead)= sum_{p>=1} phi_{m',p} R_p,   m' = floor(N/2)
// tab = [3][M] FP64 coefficient rows for these three sums.  Per chain, adds
// |L|^2, |u_m|^2, |r_m - r_cm|^2 and 1 to shape[c][0..3] and (R_p^a)^2 to
// power[c][a][p] (R_0 = sqrt(M) r_cm).  Displacements over non-overlapping
// windows of lag.v[i] samples (sample index k) of four vectors x: the centre
// of mass (FP64), the middle bead relative to it r_m' - r_cm (observable iii),
// the end-to-end vector L (observable i) and the middle bond u_m (observable
// ii): when k is a multiple of lag.v[i], adds |x - snap_i|^2 and 1 to the
// vector's window sums [c][i][0..1] from the second window edge on and sets
// snap_i = x.  For a stationary X, <X(t).X(0)> = <X^2> - <|X(t) - X(0)|^2> / 2,
// so the windows of L and u_m give their time autocorrelations.  Windows and
// snapshots are [c][kMaxLags][...] whatever lag.n is; win[v] and snp[v] hold
// vector v = 0 (centre of mass), 1 (middle bead), 2 (L), 3 (u_m).
// Bound by FP64 issue (about 60 cycles a warp instruction on a sub-partition), not by the
// 48 bytes a mode: so the warp's sums are folded rather than each summed over all
// lanes (12 additions, not 45) and a lane takes one vector and lag instead of lane 0 all of
// them (4096 chains of 64 beads, 400 steps with 20 samples: 1.84 -> 1.48 ms).
// ---------------------------------------------------------------------------
constexpr int kMaxLags = 8;         // lanes per vector of k_sample
struct SampleLags {
    int n;
    int v[kMaxLags];
};

struct SampleWindows {
    double* win[4];    // [C][kMaxLags][2] per vector
    double* snp[4];    // [C][kMaxLags][3] per vector
};

template <typename T>
__global__ void __launch_bounds__(128)
k_sample(const T* __restrict__ R, const double* __restrict__ com, const double* __restrict__ tab,
         int C, int M, double* __restrict__ shape, double* __restrict__ power, SampleWindows wv,
         int64_t k, SampleLags lag)
{
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= C) return;                 // the whole warp
    const T* Rc = R + (size_t)c * 3 * M;
    double* pw = power + (size_t)c * 3 * M;
    double s[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};      // L, u_m, r_m' - r_cm
    const double sqM = sqrt((double)M);
    for (int p = lane; p < M; p += 32) {
        const double cl = tab[p], cu = tab[M + p], cd = tab[2 * M + p];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double x = (p == 0) ? 0.0 : (double)Rc[(size_t)a * M + p];
            s[a] += cl * x;
            s[3 + a] += cu * x;
            s[6 + a] += cd * x;
            const double xp = (p == 0) ? sqM * com[3 * c + a] : x;
            pw[(size_t)a * M + p] += xp * xp;
        }
    }
    // sums over the warp: at each distance a lane keeps half of its values and hands the
    // others over (5, 3, 2, 1 of 9, then the last pair): 12 additions
    double k5[5], k3[3], k2[2];
    auto fold = [&](bool hi, double lower, double upper, int o) {
        return (hi ? upper : lower) + __shfl_xor_sync(0xffffffffu, hi ? lower : upper, o);
    };
#pragma unroll
    for (int i = 0; i < 5; ++i) k5[i] = fold(lane & 16, s[i], i < 4 ? s[5 + i] : 0.0, 16);
#pragma unroll
    for (int i = 0; i < 3; ++i) k3[i] = fold(lane & 8, k5[i], i < 2 ? k5[3 + i] : 0.0, 8);
#pragma unroll
    for (int i = 0; i < 2; ++i) k2[i] = fold(lane & 4, k3[i], i < 1 ? k3[2] : 0.0, 4);
    double t = fold(lane & 2, k2[0], k2[1], 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    // lane 8 v + i: vector v and lag i; the lanes that hold the sums of v
    const int v = lane >> 3, i = lane & 7;
    double x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        constexpr int kAt[9] = {0, 2, 4, 8, 10, 16, 18, 20, 24};
        const int at = v == 1 ? kAt[6 + a] : v == 2 ? kAt[a] : kAt[3 + a];
        x[a] = __shfl_sync(0xffffffffu, t, at);
        if (v == 0) x[a] = com[3 * c + a];
    }
    if (i == 0) {
        double* sh = shape + 4 * (size_t)c + (v == 0 ? 3 : v == 1 ? 2 : v - 2);
        *sh += v == 0 ? 1.0 : x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
    }
    if (i >= lag.n || lag.v[i] <= 0 || k % lag.v[i] != 0) return;
    const size_t w = (size_t)c * kMaxLags + i;
    double* sn = wv.snp[v] + w * 3;
    if (k > 0) {
        double d2 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double d = x[a] - sn[a];
            d2 += d * d;
        }
        wv.win[v][w * 2] += d2;
        wv.win[v][w * 2 + 1] += 1.0;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) sn[a] = x[a];
}

}  // namespace sfp

namespace sfp {

// ---------------------------------------------------------------------------
// Default bead-position Euler scheme (Sec. 3A, Eqs. b3-b5), integrated on the
// bond vectors u_n = r_n - r_{n-1} (n = 1..N; slot 0 unused) with the centre
// of mass in FP64, one block per chain, n_steps steps per launch:
//   e_n = (|u_n| - 1) u_n/|u_n| - nu (u_{n-1} + u_{n+1}),  u_0 = u_{N+1} = 0
//   bead force F_n = e_{n+1} - e_n (e_0 = e_{N+1} = 0), so the bond update is
//   u_n += dtau (e_{n+1} - 2 e_n + e_{n-1}) + a (z_n - z_{n-1}) [+ dtau g u_n^y x]
//   r_cm += a sum_n z_n / M [+ dtau g y_cm x],   a = sqrt(2 T* dtau)
// with z_n the bead normals of the mode-space path (same Philox stream).
// Shared memory: 6 M + 3 values of T (bonds, then noise; e with two zero ends).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_euler_bonds(T* __restrict__ U, double* __restrict__ com, int64_t* __restrict__ step,
                              const uint32_t* __restrict__ job, const double* __restrict__ shear,
                              int C, int M, T dtau, T amp, T nu, uint32_t seed, int n_steps,
                              int* __restrict__ bad)
{
    extern __shared__ unsigned char euler_smem[];
    T* su = reinterpret_cast<T*>(euler_smem);   // [3][M] bonds, later noise
    T* se = su + 3 * M;                          // [3][M+1] e_0 .. e_N (e_0 = 0 stays)
    __shared__ double red[3][32];
    const int c = blockIdx.x;
    if (c >= C) return;
    const int N = M - 1;
    T* Uc = U + (size_t)c * 3 * M;
    const uint32_t jb = job[c];
    const double sh = shear[c];
    int64_t st = step[c];
    bool fin = true;
    for (int s = 0; s < n_steps; ++s, ++st) {
        for (int i = threadIdx.x; i < 3 * M; i += blockDim.x) su[i] = Uc[i];
        __syncthreads();
        // e_n for bonds n = 1..N; e_0 and e_{N+1} are zero
        for (int n = threadIdx.x; n <= N + 1; n += blockDim.x) {
            T e[3] = {T(0), T(0), T(0)};
            if (n >= 1 && n <= N) {
                T u[3], um[3], up[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    u[a] = su[a * M + n];
                    um[a] = n >= 2 ? su[a * M + n - 1] : T(0);
                    up[a] = n + 1 <= N ? su[a * M + n + 1] : T(0);
                }
                const T len = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                const T f = (len - T(1)) / len;
#pragma unroll
                for (int a = 0; a < 3; ++a) e[a] = f * u[a] - nu * (um[a] + up[a]);
            }
            if (n <= N) {
#pragma unroll
                for (int a = 0; a < 3; ++a) se[a * (M + 1) + n] = e[a];
            } else {
#pragma unroll
                for (int a = 0; a < 3; ++a) se[a * (M + 1) + n] = T(0);
            }
        }
        // bonds stay in registers of the thread that updates them
        __syncthreads();
        T unew[3][4];   // up to 4 bonds per thread (M <= 4 blockDim)
        int k = 0;
        for (int n = threadIdx.x; n < M; n += blockDim.x, ++k)
#pragma unroll
            for (int a = 0; a < 3; ++a) unew[a][k] = su[a * M + n];
        __syncthreads();
        // bead noise of this step into su (the bonds are in registers now)
        double zs[3] = {0.0, 0.0, 0.0};
        for (int qd = threadIdx.x; 4 * qd < M; qd += blockDim.x) {
            T g[3][4];
            bead_quad_normals<T>(seed, jb, st, (uint32_t)qd, 0u, g);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int n = 4 * qd + i;
                if (n >= M) break;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    su[a * M + n] = g[a][i];
                    zs[a] += (double)g[a][i];
                }
            }
        }
        // block sum of the noise (centre of mass)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double v = zs[a];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 31) == 0) red[a][threadIdx.x >> 5] = v;
        }
        __syncthreads();
        k = 0;
        for (int n = threadIdx.x; n < M; n += blockDim.x, ++k) {
            if (n == 0) continue;
            T o[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const T lap = se[a * (M + 1) + n + 1] - T(2) * se[a * (M + 1) + n] + se[a * (M + 1) + n - 1];
                o[a] = unew[a][k] + dtau * lap + amp * (su[a * M + n] - su[a * M + n - 1]);
            }
            o[0] += dtau * (T)sh * unew[1][k];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                fin = fin && isfinite(o[a]);
                Uc[a * M + n] = o[a];
            }
        }
        if (threadIdx.x == 0) {
            double tot[3] = {0.0, 0.0, 0.0};
            for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w)
#pragma unroll
                for (int a = 0; a < 3; ++a) tot[a] += red[a][w];
            double* cm = com + 3 * (size_t)c;
            const double ycm = cm[1];
#pragma unroll
            for (int a = 0; a < 3; ++a) cm[a] += (double)amp * tot[a] / (double)M;
            cm[0] += (double)dtau * sh * ycm;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) step[c] = st;
    if (!fin) atomicOr(bad, 1);
}

}  // namespace sfp
