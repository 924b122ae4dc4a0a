// noise.cu -- white noise, SIMT noise filters, spectra, filter taps and the
// FP64 kappa_P solve of the QTB / QTB-PIMD random force (sm_103a).
//
// Eqs. 6-7: the random force has spectral density 2 m gamma theta(w,T);
// Eq. 12: QTB-PIMD uses kappa_P (Eq. 10) instead.  The force of the O step is
// sqrt((1-c1^2)/m) eta_n, eta_n = sum_{k=-K..K} h_|k| xi_{n-k}: a zero-phase
// time-domain filter of counter-based white noise xi whose response equals
// sqrt(S(w_j)) on the grid w_j = 2 pi j/(L dt), S = theta W or kappa_P W.
#include <cuda_bf16.h>

#include <algorithm>

#include "qtb_dev.cuh"
#include "qtb_kernels.cuh"
#include "qtb_normal.cuh"

namespace qtb {

// ---------------------------------------------------------------------------
// White noise: one Philox call per (dof, 4 steps).

template <class T> struct RingStore;
template <> struct RingStore<double> {
    __device__ static void put(double *p, double a, double b, double c, double d)
    {
        reinterpret_cast<double2 *>(p)[0] = make_double2(a, b);
        reinterpret_cast<double2 *>(p)[1] = make_double2(c, d);
    }
};
template <> struct RingStore<float> {
    __device__ static void put(float *p, float a, float b, float c, float d)
    {
        *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
    }
};
template <> struct RingStore<__nv_bfloat16> {
    __device__ static void put(__nv_bfloat16 *p, float a, float b, float c, float d)
    {
        __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t *>(&lo);
        u.y = *reinterpret_cast<uint32_t *>(&hi);
        *reinterpret_cast<uint2 *>(p) = u;
    }
};

// Generate white block `blk` (blk_abs >= -2^40; blk_override == LLONG_MIN means
// clock + Kb) into its ring slot.  grid = (ceil(max dofp * 64 / 256), nsys).
template <class T, class C>
__global__ void k_white(Dev d, long long blk_override)
{
    const DSys s = d.sys[blockIdx.y];
    long long local = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int dofl = (int)(local >> 6), qi = (int)(local & 63);
    if (dofl >= s.dofp || s.fft) return;
    long long blk = (blk_override == LLONG_MIN) ? d.clock[0] + d.Kb : blk_override;
    int slot = (int)(blk - floor_div(blk, d.nslots) * d.nslots);
    T *dst = reinterpret_cast<T *>(d.ring) + ((size_t)slot * d.Dtot + s.dof0 + dofl) * d.ring_row + 4 * qi;
    C z[4] = {0, 0, 0, 0};
    if (dofl < 3 * s.N * s.P) white4(d, blockIdx.y, dofl, blk * (kBlockSteps / 4) + qi, z);
    RingStore<T>::put(dst, z[0], z[1], z[2], z[3]);
}

// ---------------------------------------------------------------------------
// SIMT filter (short taps; longer ones: noise_fft.cu): one CTA (256 threads = 256 output steps) per dof.
// grid = (max dofp, nsys); dynamic smem = (256 + 2 Kmax + Kmax + 1) * sizeof(T)
template <class T>
__global__ void k_filter_simt(Dev d)
{
    extern __shared__ unsigned char smraw[];
    T *win = reinterpret_cast<T *>(smraw);
    const DSys s = d.sys[blockIdx.y];
    int dofl = blockIdx.x;
    if (dofl >= s.dofp || s.fft) return;
    const int K = s.K, span = kBlockSteps + 2 * K;
    T *h = win + span;
    long long blk = d.clock[0];
    T *eta = reinterpret_cast<T *>(d.eta);
    const int j = threadIdx.x;
    if (dofl >= 3 * s.N * s.P) {
        eta[(size_t)j * d.Dtot + s.dof0 + dofl] = T(0);
        return;
    }
    const T *ring = reinterpret_cast<const T *>(d.ring);
    const T *taps = reinterpret_cast<const T *>(d.tapsR) + s.taps0;
    for (int t = threadIdx.x; t < span; t += blockDim.x) {
        long long n = blk * kBlockSteps - K + t;
        long long rb = floor_div(n, kBlockSteps);
        int slot = (int)(rb - floor_div(rb, d.nslots) * d.nslots);
        win[t] = ring[((size_t)slot * d.Dtot + s.dof0 + dofl) * d.ring_row + (int)(n - rb * kBlockSteps)];
    }
    for (int t = threadIdx.x; t <= K; t += blockDim.x) h[t] = taps[t];
    __syncthreads();
    // xi(n - k) with n = blk*256 + j sits at window index j + K - k
    T acc = h[0] * win[j + K];
    for (int k = 1; k <= K; ++k) acc += h[k] * (win[j + K - k] + win[j + K + k]);
    eta[(size_t)j * d.Dtot + s.dof0 + dofl] = acc;
}

// FP32 filter of longer taps: the same sums in the same order (bit for bit) with
// their operands in registers.  A warp takes one dof, a lane 8 consecutive steps; of
// the window, which slides by one step a tap on either side, four new values a side
// come with one 16-byte load each four taps, so that 64 of ~75 instructions are the
// additions and multiply-adds themselves.  The window lies in shared memory with 4
// words of padding every 32, which puts the lanes' 16-byte loads (32 bytes apart) on
// different banks.  Measured, 262152 dofs, 2049 taps: 6.4 ms a
// block instead of 19.5 (k_filter_simt); its instructions alone would take 4.3.
constexpr int kTileDofs = 8;   // dofs (warps) per CTA: full 32-byte sectors of eta
constexpr int kTileTaps = 16;  // taps per loop iteration (the register windows rotate in place)
__host__ __device__ constexpr int tile_taps(int K) { return (K + kTileTaps) / kTileTaps * kTileTaps; }  // 0 .. K, rounded up
__host__ __device__ constexpr int tile_pad(int i) { return i + 4 * (i >> 5); }
// words of a window: the steps, 16 of margin a side for the zeros past tap K, alignment
__host__ __device__ constexpr int tile_window(int K) { return (tile_pad(kBlockSteps + 2 * K + 48) + 7) & ~3; }

__global__ void __launch_bounds__(32 * kTileDofs) k_filter_tile(Dev d, int Kmax)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const DSys s = d.sys[blockIdx.y];
    const int dof0 = blockIdx.x * kTileDofs;
    if (dof0 >= s.dofp) return;
    const int K = s.K, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, dofl = dof0 + warp;
    float *h = reinterpret_cast<float *>(smraw);         // taps, h_0 and those past K as zeros
    float *win = h + tile_taps(Kmax) + (size_t)warp * tile_window(Kmax);
    // step blk 256 + i - K at window index o + i: o + K mod 4 = 3 aligns the loads below
    const int o = 16 + ((3 - K) & 3), span = kBlockSteps + 2 * K;
    const float *ring = reinterpret_cast<const float *>(d.ring);
    const float *taps = reinterpret_cast<const float *>(d.tapsR) + s.taps0;
    const long long blk = d.clock[0];
    for (int t = threadIdx.x; t < tile_taps(K); t += blockDim.x) h[t] = t > 0 && t <= K ? taps[t] : 0.0f;
    for (int q = -d.Kb; q <= d.Kb; ++q) {
        const long long rb = blk + q;
        const int slot = (int)(rb - floor_div(rb, d.nslots) * d.nslots);
        const float *src = ring + ((size_t)slot * d.Dtot + s.dof0 + dofl) * d.ring_row;
        for (int e = lane; e < kBlockSteps; e += 32) {
            const int i = q * kBlockSteps + K + e;
            if (i >= 0 && i < span) win[tile_pad(o + i)] = src[e];
        }
    }
    // the margins that the zeros past tap K meet
    if (lane < o) win[tile_pad(lane)] = 0.0f;
    if (lane < 16) win[tile_pad(o + span + lane)] = 0.0f;
    __syncthreads();
    const int c = o + 8 * lane + K;  // window index of this lane's first step; c mod 4 = 3
    // Blocks of four window values: block m of the left side starts at c - 3 - 4 m, of the
    // right side at c - 3 + 4 m.  Taps 4 m .. 4 m + 3 meet the left blocks m, m - 1, m - 2
    // and the right ones m .. m + 3; block m lives in slot m mod 4.
    float acc[8], L[4][4], Rw[4][4];
    auto load4 = [&](int i, float (&r)[4]) {
        const float4 v = *reinterpret_cast<const float4 *>(win + tile_pad(i));
        r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
    };
    load4(c - 3 + 4, L[3]);
    load4(c - 3 + 8, L[2]);
#pragma unroll
    for (int m = 0; m < 3; ++m) load4(c - 3 + 4 * m, Rw[m]);
    const float h0 = taps[0];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = h0 * Rw[(i + 3) >> 2][(i + 3) & 3];
    for (int k0 = 0; k0 <= K; k0 += kTileTaps) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            load4(c - 3 - k0 - 4 * m, L[m]);
            load4(c - 3 + k0 + 4 * (m + 3), Rw[(m + 3) & 3]);
            const float4 hv = *reinterpret_cast<const float4 *>(h + k0 + 4 * m);
            const float hk[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int l = i + 3 - k, r = i + 3 + k;
                    acc[i] = fmaf(hk[k], L[(m - (l >> 2)) & 3][l & 3] + Rw[(m + (r >> 2)) & 3][r & 3], acc[i]);
                }
        }
    }
    // steps by rows of the CTA's dofs
    __syncthreads();
    float *rows = h;  // [256][kTileDofs + 1]
    const bool real = dofl < 3 * s.N * s.P;
#pragma unroll
    for (int i = 0; i < 8; ++i) rows[(8 * lane + i) * (kTileDofs + 1) + warp] = real ? acc[i] : 0.0f;
    __syncthreads();
    float *eta = reinterpret_cast<float *>(d.eta) + s.dof0 + dof0;
    for (int e = threadIdx.x; e < kBlockSteps * kTileDofs; e += blockDim.x) {
        const int j = e / kTileDofs, l = e % kTileDofs;
        eta[(size_t)j * d.Dtot + l] = rows[j * (kTileDofs + 1) + l];
    }
}

static size_t tile_smem(int Kmax)
{
    const size_t w = (size_t)tile_taps(Kmax) + (size_t)kTileDofs * tile_window(Kmax);
    return 4 * std::max(w, (size_t)kBlockSteps * (kTileDofs + 1));
}

// ---------------------------------------------------------------------------
// Spectra and taps (FP64).

__device__ double theta_dev(double w, double T)
{
    w = fabs(w);
    double kT = kBoltz * T;
    double x = kHbar * w / kT;
    if (x < 1e-6) return kT * (1.0 + x * x / 12.0);
    return kHbar * w * (0.5 + 1.0 / expm1(x));
}

__device__ double fth_dev(double x)
{
    x = fabs(x);
    if (x < 1e-6) return 1.0 + x * x / 12.0;
    return x * (0.5 + 1.0 / expm1(x));
}

__device__ double kappa_tail_dev(int P, double y)
{
    if (P == 1) return fth_dev(y);
    return fth_dev(sqrt((double)P) * y) / P + sqrt((double)P) / (2.0 * y);
}

// F_P at y from the collocation grid y_i = y0 sinh(i dts)
__device__ double kappa_eval_dev(const DSpec &sp, double y)
{
    if (sp.P == 1) return fth_dev(y);
    if (y > sp.ymax) return kappa_tail_dev(sp.P, y);
    double dts = asinh(sp.ymax / sp.y0) / (sp.n - 1);
    int i = (int)(asinh(y / sp.y0) / dts);
    if (i > sp.n - 2) i = sp.n - 2;
    double ya = sp.y0 * sinh(i * dts), yb = sp.y0 * sinh((i + 1) * dts);
    double lam = (y - ya) / (yb - ya);
    return sp.F[i] * (1.0 - lam) + sp.F[i + 1] * lam;
}

// S_j, j = 0..K, per system.  grid = (ceil((Kmax+1)/256), nsys)
// spectral density at w (rad/fs) of a system in a non-learned mode: k_B T
// (white), theta (QTB, Eq. 7) or kappa_P (QTB-PIMD, Eq. 12), times the cutoff
__device__ double spectrum_value(const DSpec &sp, double w)
{
    double base;
    if (sp.mode == QTB_NOISE_WHITE) {
        base = kBoltz * sp.T;
    } else if (sp.mode == QTB_NOISE_QTB) {
        base = theta_dev(w, sp.T);
    } else {
        double kT = kBoltz * sp.T;
        base = kT * kappa_eval_dev(sp, kHbar * w / kT);
    }
    double W = 1.0;
    if (sp.mode != QTB_NOISE_WHITE && sp.omega_max > 0.0)
        W = 1.0 / (1.0 + exp((w - sp.omega_max) / (sp.omega_max / 50.0)));
    return base * W;
}

__global__ void k_spectrum(const DSpec *spec, double *S)
{
    const DSpec sp = spec[blockIdx.y];
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > sp.K) return;
    if (sp.mode == QTB_NOISE_QTB_PIMD_MLP) return;  // filled by the learned model's spectrum kernel (mlp.cu)
    int L = 2 * sp.K + 1;
    S[sp.taps0 + j] = spectrum_value(sp, 2.0 * kPi * j / (L * sp.dt));
}

// sqrt(S_j) in place and the table cos(2 pi j/L), j = 0..K (the cosine transform's
// square roots and cosines, once each instead of once per tap: K^2 of either took 2 ms
// of the FP64 pipes at K = 1024, now 0.1 ms)
__global__ void k_taps_table(const DSpec *spec, double *S, double *cs)
{
    const DSpec sp = spec[blockIdx.y];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > sp.K) return;
    S[sp.taps0 + j] = sqrt(S[sp.taps0 + j]);
    cs[sp.taps0 + j] = cospi(2.0 * (double)j / (double)(2 * sp.K + 1));
}

__global__ void k_taps(const DSpec *spec, const double *S, const double *cs, double *h64, float *h32)
{
    const DSpec sp = spec[blockIdx.y];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > sp.K) return;
    const int K = sp.K, L = 2 * K + 1;
    const double *Sj = S + sp.taps0, *cj = cs + sp.taps0;
    double acc = 0.0;
    int m = 0;  // j k mod L
    for (int j = 1; j <= K; ++j) {
        m += k;
        if (m >= L) m -= L;
        acc += Sj[j] * cj[min(m, L - m)];
    }
    const double h = (Sj[0] + 2.0 * acc) / (double)L;
    h64[sp.taps0 + k] = h;
    h32[sp.taps0 + k] = (float)h;
}

// ---------------------------------------------------------------------------
// kappa_P solve (Eq. 10), FP64: collocation rows, normal equations, blocked Cholesky,
// triangular solves, one refinement step.
//
// A row has 2 P nonzeros on its P curves y_k(y), and the curves run together at large y:
// of the 32 x 32 tiles of A most are zero, and the normal matrix is dense only in its
// leading part (columns up to asinh sqrt(4 P)) and narrow-banded beyond.  Everything
// below works on tiles and skips the zero ones (what they would add is exactly zero):
// flags per tile of A, and per tile row of the factor the first nonzero tile
// (Cholesky keeps that envelope).  One solve (P = 8, n = 1024): 3.0 ms; with dense
// normal equations, one-warp panels and unblocked triangular solves 17.5.
constexpr int kCholNb = 32;

static inline int kappa_words(int n) { return ((n + kCholNb - 1) / kCholNb + 31) / 32; }  // flag words per tile row of A
// envelope of the factor: ints in row 0 of M from column 32 on (the strict upper triangle
// of M is not used outside the diagonal tiles; one tile has no envelope)
__device__ __forceinline__ int *kappa_env(double *M) { return reinterpret_cast<int *>(M + kCholNb); }
__device__ __forceinline__ const int *kappa_env(const double *M) { return reinterpret_cast<const int *>(M + kCholNb); }

struct KappaTerm {
    double w, lam;  // weight; position in the interval, or (i < 0) the tail's value
    int i;          // left node of the interval, -1: beyond the grid, -2: no term
};
__device__ __forceinline__ KappaTerm kappa_term(int P, int n, double ymax, double y0, double dts, int m, int k)
{
    const double y = y0 * sinh(0.5 * m * dts), sk = sinpi((double)k / P), ck = 4.0 * P * sk * sk, yk = sqrt(y * y + ck);
    KappaTerm t;
    t.w = (k == 0) ? 1.0 : ((y * y + ck) > 0.0 ? y * y / (y * y + ck) : 0.0);
    t.lam = 0.0;
    t.i = -2;
    if (t.w == 0.0) return t;
    if (yk <= ymax) {
        t.i = min((int)(asinh(yk / y0) / dts), n - 2);
        const double ya = y0 * sinh(t.i * dts), yb = y0 * sinh((t.i + 1) * dts);
        t.lam = (yk - ya) / (yb - ya);
    } else {
        t.i = -1;
        t.lam = kappa_tail_dev(P, yk);
    }
    return t;
}

// the terms of every row (their inverse hyperbolic functions are most of the work), one
// thread each; grid = (ceil(rows / 128), P)
__global__ void k_kappa_terms(int P, int n, double ymax, double y0, KappaTerm *t)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (m < 2 * n - 1) t[(size_t)m * P + k] = kappa_term(P, n, ymax, y0, asinh(ymax / y0) / (n - 1), m, k);
}

// rows m < 2n-1 from their terms (null: formed here), unscaled; A is (2n-1) x n row-major,
// zeroed by the caller; b[m] and, for k_kappa_scale, sc[m] = 1/f
__global__ void k_kappa_rows(int P, int n, double ymax, double y0, const KappaTerm *terms, double *A, double *b, double *sc)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= 2 * n - 1) return;
    const double dts = asinh(ymax / y0) / (n - 1), y = y0 * sinh(0.5 * m * dts);
    const double f = fth_dev(sqrt((double)P) * y);
    double rhs = f;
    double *Ar = A + (size_t)m * n;
    for (int k = 0; k < P; ++k) {
        const KappaTerm t = terms ? terms[(size_t)m * P + k] : kappa_term(P, n, ymax, y0, dts, m, k);
        if (t.i >= 0) {
            Ar[t.i] += t.w * (1.0 - t.lam);
            Ar[t.i + 1] += t.w * t.lam;
        } else if (t.i == -1) {
            rhs -= t.w * t.lam;
        }
    }
    sc[m] = 1.0 / f;
    b[m] = rhs * (1.0 / f);
}

// rows times sc, and the flags of their nonzero tiles; one CTA of 256 per 32 rows
__global__ void k_kappa_scale(int n, const double *sc, double *A, unsigned *nz, int words)
{
    const int m0 = blockIdx.x * kCholNb, rows = 2 * n - 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int ct = warp; ct * kCholNb < n; ct += 8) {
        const int i = ct * kCholNb + lane;
        bool any = false;
        for (int q = 0; q < kCholNb; ++q) {
            const int m = m0 + q;
            if (m < rows && i < n) {
                const double a = A[(size_t)m * n + i];
                if (a != 0.0) {
                    any = true;
                    A[(size_t)m * n + i] = a * sc[m];
                }
            }
        }
        if (__any_sync(0xffffffffu, any) && lane == 0 && nz) atomicOr(&nz[blockIdx.x * words + (ct >> 5)], 1u << (ct & 31));
    }
}

// envelope: first tile column tj with a nonzero tile (ti, tj) of M = A^T A, per tile
// row; one CTA per ti, one thread per tile row of A
__global__ void k_kappa_envelope(int n, const unsigned *nz, int words, double *M)
{
    __shared__ int first;
    const int ti = blockIdx.x, nmt = (2 * n - 1 + kCholNb - 1) / kCholNb;
    if (threadIdx.x == 0) first = nz ? ti : 0;
    __syncthreads();
    for (int mt = threadIdx.x; nz && mt < nmt; mt += blockDim.x)
        if ((nz[mt * words + (ti >> 5)] >> (ti & 31)) & 1u)
            for (int w = 0; w < words; ++w)
                if (nz[mt * words + w]) {
                    atomicMin(&first, 32 * w + __ffs(nz[mt * words + w]) - 1);
                    break;
                }
    __syncthreads();
    if (threadIdx.x == 0) kappa_env(M)[ti] = first;
}

// M = A^T A, lower triangle, over the tile rows of A that meet both tile columns;
// blockIdx.x enumerates the tiles (ti >= tj); 256 threads, each 4 outputs
__global__ void k_kappa_normal(int n, const double *A, const unsigned *nz, int words, double *M)
{
    __shared__ double ta[32][33], tb[32][33];
    int tj = blockIdx.x, ti = 0;
    while (tj > ti) { tj -= ti + 1; ++ti; }
    const int rows = 2 * n - 1, nmt = (rows + kCholNb - 1) / kCholNb;
    const int i0 = ti * 32, j0 = tj * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // ty in 0..7
    double acc[4] = {0, 0, 0, 0};
    for (int mt = 0; mt < nmt; ++mt) {
        if (nz) {
            const unsigned fi = nz[mt * words + (ti >> 5)] >> (ti & 31), fj = nz[mt * words + (tj >> 5)] >> (tj & 31);
            if (!(fi & fj & 1u)) continue;  // uniform over the CTA
        }
        const int m0 = mt * kCholNb;
        for (int q = 0; q < 4; ++q) {
            const int mm = m0 + ty + 8 * q;
            ta[ty + 8 * q][tx] = (mm < rows && i0 + tx < n) ? A[(size_t)mm * n + i0 + tx] : 0.0;
            tb[ty + 8 * q][tx] = (mm < rows && j0 + tx < n) ? A[(size_t)mm * n + j0 + tx] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int mm = 0; mm < 32; ++mm)
            for (int q = 0; q < 4; ++q) acc[q] += ta[mm][ty + 8 * q] * tb[mm][tx];
        __syncthreads();
    }
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + ty + 8 * q, j = j0 + tx;
        if (i < n && j < n) M[(size_t)i * n + j] = acc[q];
    }
}

// g = A^T s; one CTA of 8 warps per 32 columns, the warps' sums added in warp order
__global__ void k_kappa_atv(int n, const double *A, const double *s, double *g)
{
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane, rows = 2 * n - 1;
    double acc = 0.0;
    if (i < n) {
#pragma unroll 8
        for (int m = warp; m < rows; m += 8) acc += A[(size_t)m * n + i] * s[m];
    }
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && i < n) {
        for (int w = 1; w < 8; ++w) acc += part[w][lane];
        g[i] = acc;
    }
}

// Blocked right-looking Cholesky of the lower triangle of M (n x n, row-major), panels
// of kCholNb columns, two launches a panel.  A warp's FP64 instruction holds its quarter
// of the SM for ~64 cycles, so a 32 x 32 block is spread over four warps, a row over
// four lanes (columns c = g mod 4); the diagonal block is eliminated without square
// roots (they follow for all rows at once).  Every CTA that needs its factor forms it
// again, which costs less than a launch in between.  (One warp with a row a lane took 85
// us a panel.)  A non-positive pivot sets ERR_SOLVE (the solve then continues on a
// placeholder pivot).  A block of at most 8 columns ends after 8: on the smallest grid, of 8
// nodes, all 32 made a solve slower than the form before (P = 2: 0.27 ms, 0.23 before and now).
constexpr int kCholThreads = 4 * kCholNb;

// 1/v: two Newton steps from the FP32 value where that is in range, else the quotient
__device__ __forceinline__ double fast_rcp(double v)
{
    if (!(v > 1e-30 && v < 1e30)) return 1.0 / v;
    double y = (double)(1.0f / (float)v);
#pragma unroll
    for (int k = 0; k < 2; ++k) y = fma(y, fma(-v, y, 1.0), y);
    return y;
}

struct CholSmem {
    double L[kCholNb][kCholNb + 1];  // L[c][r]: column c of the factor (r > c)
    double rd[kCholNb];              // reciprocals of its diagonal
    double col[2][kCholNb];
};

// factor of the block at (k0, k0) into B, by threads 0 .. kCholThreads - 1 of a CTA whose
// threads all call it
__device__ __forceinline__ void chol_factor32(int n, int k0, const double *M, CholSmem &B, unsigned *err)
{
    const int t = threadIdx.x, r = t >> 2, g = t & 3;
    const bool mine = t < kCholThreads;
    double a[kCholNb / 4];
#pragma unroll
    for (int q = 0; q < kCholNb / 4; ++q) {
        const int c = 4 * q + g;
        a[q] = mine && k0 + r < n && c <= r ? M[(size_t)(k0 + r) * n + k0 + c] : (c == r ? 1.0 : 0.0);
    }
#pragma unroll
    for (int j = 0; j < kCholNb; ++j) {
        if (j == 8 && k0 + 8 >= n) break;  // the smallest grids: the rest is the identity (uniform)
        double *col = B.col[j & 1];
        if (mine && g == (j & 3)) col[r] = a[j / 4];
        __syncthreads();
        if (mine && r >= j) {
            double v = col[j];
            if (!(v > 0.0)) {
                if (r == j && g == 0 && err) atomicOr(err, (unsigned)ERR_SOLVE);
                v = 1e-300;
            }
            const double x = col[r];
            if (g == 0) {
                if (r == j) B.rd[j] = v;
                else B.L[j][r] = x;
            }
            if (r > j) {
                const double f = x * fast_rcp(v);
#pragma unroll
                for (int q = j / 4; q < kCholNb / 4; ++q)
                    if (4 * q + g > j) a[q] = fma(-f, col[4 * q + g], a[q]);  // (columns past r stay unused)
            }
        }
    }
    __syncthreads();
    if (t < kCholNb) B.rd[t] = rsqrt(B.rd[t]);
    __syncthreads();
    if (mine)
        for (int c = g; c < r; c += 4) B.L[c][r] *= B.rd[c];
    __syncthreads();
}

// rows r0 = k0 + 32 (1 + blockIdx.x) .. (+32) of the panel: X L11^T = A21
__global__ void __launch_bounds__(kCholThreads) k_chol_panel(int n, int k0, double *M)
{
    __shared__ CholSmem B;
    const int ti = k0 / kCholNb + 1 + blockIdx.x;
    if (kappa_env(M)[ti] > k0 / kCholNb) return;  // zero rows (uniform over the CTA)
    chol_factor32(n, k0, M, B, nullptr);
    const int t = threadIdx.x, g = t & 3, r = ti * kCholNb + (t >> 2);
    double a[kCholNb / 4];
#pragma unroll
    for (int q = 0; q < kCholNb / 4; ++q) a[q] = r < n ? M[(size_t)r * n + k0 + 4 * q + g] : 0.0;
#pragma unroll
    for (int j = 0; j < kCholNb; ++j) {
        const double x = __shfl_sync(0xffffffffu, a[j / 4], j & 3, 4) * B.rd[j];
        if (g == (j & 3)) a[j / 4] = x;
#pragma unroll
        for (int q = j / 4; q < kCholNb / 4; ++q)
            if (4 * q + g > j) a[q] = fma(-x, B.L[j][4 * q + g], a[q]);
    }
    if (r < n)
#pragma unroll
        for (int q = 0; q < kCholNb / 4; ++q) M[(size_t)r * n + k0 + 4 * q + g] = a[q];
}

// trailing update below the panel, blockIdx.x - 1 enumerating the tiles (ti >= tj) of the
// trailing matrix; block 0 stores the diagonal block's factor (read unfactored by the
// panel's CTAs before) the way the triangular solves take it: reciprocal diagonal rd,
// below it L_ij rd_j, above it L_ji rd_j
__global__ void __launch_bounds__(256) k_chol_update(int n, int k0, double *M, unsigned *err)
{
    __shared__ union {
        CholSmem B;
        double L[2][kCholNb][kCholNb + 1];
    } sm;
    if (blockIdx.x == 0) {
        chol_factor32(n, k0, M, sm.B, err);
        for (int e = threadIdx.x; e < kCholNb * kCholNb; e += blockDim.x) {
            const int r = e / kCholNb, c = e % kCholNb;
            if (k0 + r < n && k0 + c < n)
                M[(size_t)(k0 + r) * n + k0 + c] = r == c ? sm.B.rd[r] : r > c ? sm.B.L[c][r] * sm.B.rd[c] : sm.B.L[r][c] * sm.B.rd[c];
        }
        return;
    }
    double (*Li)[kCholNb + 1] = sm.L[0], (*Lj)[kCholNb + 1] = sm.L[1];
    int tj = blockIdx.x - 1, ti = 0;
    while (tj > ti) { tj -= ti + 1; ++ti; }
    const int kt = k0 / kCholNb;
    ti += kt + 1;
    tj += kt + 1;
    if (kappa_env(M)[ti] > kt || kappa_env(M)[tj] > kt) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, ri0 = ti * kCholNb, rj0 = tj * kCholNb;
    for (int q = ty; q < kCholNb; q += 8) {
        Li[q][tx] = ri0 + q < n ? M[(size_t)(ri0 + q) * n + k0 + tx] : 0.0;
        Lj[q][tx] = rj0 + q < n ? M[(size_t)(rj0 + q) * n + k0 + tx] : 0.0;
    }
    __syncthreads();
    double acc[4] = {0, 0, 0, 0};
#pragma unroll 8
    for (int e = 0; e < kCholNb; ++e)
        for (int q = 0; q < 4; ++q) acc[q] += Li[ty + 8 * q][e] * Lj[tx][e];
    for (int q = 0; q < 4; ++q) {
        const int i = ri0 + ty + 8 * q, j = rj0 + tx;
        if (i < n && j <= i) M[(size_t)i * n + j] -= acc[q];
    }
}

static void chol_blocked(int n, double *M, unsigned *err, cudaStream_t st)
{
    for (int k0 = 0; k0 < n; k0 += kCholNb) {
        const int nt = std::max(0, (n - k0 - 1) / kCholNb);  // tile rows below
        if (nt) k_chol_panel<<<nt, kCholThreads, 0, st>>>(n, k0, M);
        k_chol_update<<<1 + nt * (nt + 1) / 2, 256, 0, st>>>(n, k0, M, err);
    }
}

// Solve L L^T x = r in place (x overwrites r), one CTA of 16 warps, block by block: the
// warps gather what the solved blocks contribute (a tile each, within the envelope),
// warp 0 adds that up in warp order and solves the block's triangle, whose entries come
// scaled (k_chol_update): a step of that chain is one broadcast and one multiply-add.
constexpr int kTrsvWarps = 16;
__global__ void __launch_bounds__(32 * kTrsvWarps) k_kappa_trsv(int n, const double *M, double *r)
{
    __shared__ double part[kTrsvWarps][kCholNb], D[kCholNb][kCholNb + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nt = (n + kCholNb - 1) / kCholNb;
    const int *env = kappa_env(M);
    for (int pass = 0; pass < 2; ++pass) {  // 0: L y = r, 1: L^T x = y
        for (int s = 0; s < nt; ++s) {
            const int kt = pass ? nt - 1 - s : s, k0 = kt * kCholNb;
            for (int q = warp; q < kCholNb; q += kTrsvWarps)
                D[q][lane] = (k0 + q < n && k0 + lane < n) ? M[(size_t)(k0 + q) * n + k0 + lane] : (q == lane ? 1.0 : 0.0);
            double acc = 0.0;
            const int t0 = pass ? kt + 1 : (nt > 1 ? env[kt] : 0), t1 = pass ? nt : kt;
            if (pass == 0) {
                const int row = k0 + lane;
                for (int tj = t0 + warp; tj < t1; tj += kTrsvWarps)
                    if (row < n) {
                        const double *Lr = M + (size_t)row * n + tj * kCholNb;
#pragma unroll 16
                        for (int e = 0; e < kCholNb; ++e) acc = fma(Lr[e], r[tj * kCholNb + e], acc);
                    }
            } else {
                const int col = k0 + lane;
                for (int ti = t0 + warp; ti < t1; ti += kTrsvWarps)
                    if (env[ti] <= kt && col < n) {
                        const int e1 = min(kCholNb, n - ti * kCholNb);
#pragma unroll 16
                        for (int e = 0; e < e1; ++e) acc = fma(M[(size_t)(ti * kCholNb + e) * n + col], r[ti * kCholNb + e], acc);
                    }
            }
            part[warp][lane] = acc;
            __syncthreads();
            if (warp == 0) {
                double x = k0 + lane < n ? r[k0 + lane] : 0.0;
                for (int w = 0; w < min(kTrsvWarps, t1 - t0); ++w) x -= part[w][lane];
                double l[kCholNb];
#pragma unroll
                for (int j = 0; j < kCholNb; ++j) l[j] = (pass == 0 ? j < lane : j > lane) ? D[lane][j] : 0.0;
                const bool more = n - k0 > 8;  // (8 columns or fewer: the rest is the identity)
                if (pass == 0) {
#pragma unroll
                    for (int j = 0; j < kCholNb; ++j) {
                        if (j == 8 && !more) break;
                        x = fma(-l[j], __shfl_sync(0xffffffffu, x, j), x);
                    }
                } else {
                    if (more)
#pragma unroll
                        for (int j = kCholNb - 1; j >= 8; --j) x = fma(-l[j], __shfl_sync(0xffffffffu, x, j), x);
#pragma unroll
                    for (int j = 7; j >= 0; --j) x = fma(-l[j], __shfl_sync(0xffffffffu, x, j), x);
                }
                if (k0 + lane < n) r[k0 + lane] = x * D[lane][lane];
            }
            __syncthreads();
        }
    }
}

// Refinement of the least-squares solution (corrected semi-normal equations,
// Bjorck): s = b - A x, g = A^T s, solve L L^T d = g with the Cholesky factor
// already in M, x += d.  The normal equations alone leave an error of order
// cond(A)^2 eps; each refinement step brings it towards cond(A) eps, the
// accuracy of an orthogonal-factorisation solve.

// s[m] = b[m] - A[m,:] x; one warp per row
__global__ void k_kappa_resid(int rows, int n, const double *A, const double *b, const double *x, double *s)
{
    const int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (m >= rows) return;
    const double *Ar = A + (size_t)m * n;
    double acc = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double a = Ar[i];
        if (a != 0.0) acc += a * x[i];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) s[m] = b[m] - acc;
}

__global__ void k_kappa_add(int n, double *x, const double *d)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] += d[i];
}

// ---------------------------------------------------------------------------
// Fourier-segment generator (Eq. 9): segments of n = 256 M steps per dof,
// eta_t = (1/sqrt(n)) sum_j c_j e^{+2 pi i j t/n}, c_0 = sqrt(S_0) xi_0,
// c_{n/2} = sqrt(S_{n/2}) xi_1, c_j = sqrt(S_j/2) (xi_2j + i xi_2j+1) and
// c_{n-j} = conj(c_j), xi the white stream of the dof over the segment.

// sqrt(S_j / n) on w_j = 2 pi j/(n dt), j = 0..n/2, per system
template <class R>
__global__ void k_spectrum_seg(const DSpec *spec, int n, R *sq)
{
    const DSpec sp = spec[blockIdx.y];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > n / 2) return;
    sq[(size_t)blockIdx.y * (n / 2 + 1) + j] = (R)sqrt(spectrum_value(sp, 2.0 * kPi * j / (n * sp.dt)) / n);
}

constexpr int kSegPairs = 2;  // dof pairs per CTA of the segment generator

// One CTA per kSegPairs pairs of dofs of one system: the n normals of each dof
// (the white stream over the segment's steps), the spectrum W = Z_a + i Z_b of a
// pair (both Z Hermitian, so the inverse transform of W carries the two real
// sequences as its real and imaginary parts), a radix-2 Stockham inverse FFT
// in shared memory (ping-pong between two buffers), eta rows t = 0..n-1.
// Launched for every block; it generates only at the first block of a segment
// unless `force`.  grid = (ceil(max dofp / (2 kSegPairs)), nsys), 256 threads,
// dynamic smem 2 kSegPairs * 2 n * sizeof(R).
template <class R, class C>
__global__ void __launch_bounds__(256) k_fourier(Dev d, const R *sq, const R *tw, int n, int force)
{
    extern __shared__ __align__(16) unsigned char fsm[];
    const long long blk = d.clock[0];
    const int M = n / kBlockSteps;
    const long long seg = floor_div(blk, M);
    if (!force && blk != seg * M) return;
    const DSys S = d.sys[blockIdx.y];
    const int dof_first = blockIdx.x * 2 * kSegPairs;
    if (dof_first >= S.dofp) return;
    const int nreal = 3 * S.N * S.P, h = n / 2;
    const size_t span = (size_t)2 * n;  // one pair's complex sequence
    R *bufA = reinterpret_cast<R *>(fsm);
    R *bufB = bufA + kSegPairs * span;
    // 1) normals: pair p, dof a (0) or b (1), step t -> bufB[p span + ab n + t]
    const int nq = n / 4;
    for (int w = threadIdx.x; w < kSegPairs * 2 * nq; w += blockDim.x) {
        const int q = w % nq, ab = (w / nq) & 1, p = w / (2 * nq);
        const int dofl = dof_first + 2 * p + ab;
        C z[4] = {0, 0, 0, 0};
        if (dofl < nreal) white4(d, blockIdx.y, dofl, seg * nq + q, z);
        R *dst = bufB + p * span + ab * n + 4 * q;
        dst[0] = (R)z[0]; dst[1] = (R)z[1]; dst[2] = (R)z[2]; dst[3] = (R)z[3];
    }
    __syncthreads();
    // 2) W_j = Z_a,j + i Z_b,j (sq holds sqrt(S_j/n): the 1/sqrt(n) is folded in)
    const R *sqs = sq + (size_t)blockIdx.y * (h + 1);
    for (int w = threadIdx.x; w < kSegPairs * n; w += blockDim.x) {
        const int j = w % n, p = w / n;
        const R *xa = bufB + p * span, *xb = xa + n;
        R re, im;
        if (j == 0) {
            re = sqs[0] * xa[0]; im = sqs[0] * xb[0];
        } else if (j == h) {
            re = sqs[h] * xa[1]; im = sqs[h] * xb[1];
        } else {
            const int jj = j < h ? j : n - j;
            const R r = sqs[jj] * (R)0.70710678118654752440;
            const R ar = xa[2 * jj], ai = xa[2 * jj + 1], br = xb[2 * jj], bi = xb[2 * jj + 1];
            if (j < h) { re = r * (ar - bi); im = r * (ai + br); }  // r (a_re + i a_im) + i r (b_re + i b_im)
            else { re = r * (ar + bi); im = r * (br - ai); }        // the conjugates
        }
        bufA[p * span + 2 * j] = re;
        bufA[p * span + 2 * j + 1] = im;
    }
    __syncthreads();
    // 3) sum_j W_j e^{+2 pi i j t/n}: stage (l, m) maps x[k + jj m], x[k + jj m + l m] to
    //    y[k + 2 jj m] = sum, y[k + 2 jj m + m] = e^{+2 pi i jj m/n} (difference)
    R *x = bufA, *y = bufB;
    for (int l = h, m = 1; l >= 1; l >>= 1, m <<= 1) {
        for (int w = threadIdx.x; w < kSegPairs * h; w += blockDim.x) {
            const int b = w % h, p = w / h;
            const int jj = b / m, k = b - jj * m;
            const R wr = tw[2 * (jj * m)], wi = tw[2 * (jj * m) + 1];
            const R *xp = x + p * span;
            R *yp = y + p * span;
            const int i0 = k + jj * m, i1 = i0 + l * m, o0 = k + 2 * jj * m, o1 = o0 + m;
            const R c0r = xp[2 * i0], c0i = xp[2 * i0 + 1], c1r = xp[2 * i1], c1i = xp[2 * i1 + 1];
            const R dr = c0r - c1r, di = c0i - c1i;
            yp[2 * o0] = c0r + c1r;
            yp[2 * o0 + 1] = c0i + c1i;
            yp[2 * o1] = fma(wr, dr, -wi * di);
            yp[2 * o1 + 1] = fma(wr, di, wi * dr);
        }
        __syncthreads();
        R *t = x;
        x = y;
        y = t;
    }
    // 4) eta rows of the segment (padding dofs: 0)
    R *eta = reinterpret_cast<R *>(d.eta);
    for (int w = threadIdx.x; w < kSegPairs * 2 * n; w += blockDim.x) {
        const int ab = w % 2, t = (w / 2) % n, p = w / (2 * n);
        const int dofl = dof_first + 2 * p + ab;
        if (dofl >= S.dofp) continue;
        eta[(size_t)t * d.Dtot + S.dof0 + dofl] = (dofl < nreal) ? x[p * span + 2 * t + ab] : R(0);
    }
}

// ---------------------------------------------------------------------------
// launchers

void launch_white(const Dev &d, int filter_kind, int max_dofp, int nsys, long long blk, cudaStream_t st)
{
    dim3 grid((unsigned)(((long long)max_dofp * 64 + 255) / 256), (unsigned)nsys);
    if (filter_kind == FK_FP64)
        k_white<double, double><<<grid, 256, 0, st>>>(d, blk);
    else if (filter_kind == FK_FP32)
        k_white<float, float><<<grid, 256, 0, st>>>(d, blk);
    else
        k_white<__nv_bfloat16, float><<<grid, 256, 0, st>>>(d, blk);
}

// the tiled FP32 filter from this half length on (below, the window loads dominate
// either form), up to what its 8 windows need of shared memory.  Measured, 32769 dofs, ms
// per 256 steps (steps included), one dof a CTA / tiled: K = 8 0.36 / 0.31, 32 0.40 / 0.33,
// 128 0.61 / 0.40, 1024 2.71 / 1.09.
constexpr int kTileMinK = 8;
constexpr size_t kTileMaxSmem = 220 * 1024;

void launch_filter_simt(const Dev &d, int filter_kind, int max_dofp, int nsys, int Kmax, cudaStream_t st)
{
    dim3 grid((unsigned)max_dofp, (unsigned)nsys);
    if (filter_kind == FK_FP64) {
        size_t sm = sizeof(double) * (kBlockSteps + 3 * Kmax + 1);
        k_filter_simt<double><<<grid, kBlockSteps, sm, st>>>(d);
    } else {
        size_t sm = sizeof(float) * (kBlockSteps + 3 * Kmax + 1);
        if (Kmax >= kTileMinK && tile_smem(Kmax) <= kTileMaxSmem)
            k_filter_tile<<<dim3((unsigned)(max_dofp / kTileDofs), (unsigned)nsys), 32 * kTileDofs, tile_smem(Kmax), st>>>(d, Kmax);
        else
            k_filter_simt<float><<<grid, kBlockSteps, sm, st>>>(d);
    }
}

cudaError_t filter_simt_prepare(int Kmax)
{
    const size_t taps = kBlockSteps + 3 * (size_t)Kmax + 1;
    cudaError_t e = allow_dynamic_smem(k_filter_simt<double>, sizeof(double) * taps);
    if (e == cudaSuccess) e = allow_dynamic_smem(k_filter_tile, std::min(tile_smem(Kmax), kTileMaxSmem));
    if (e == cudaSuccess) e = allow_dynamic_smem(k_filter_simt<float>, sizeof(float) * taps);
    return e;
}

void launch_spectrum_taps(const DSpec *spec, int nsys, int Kmax, double *S, double *cs, double *h64, float *h32,
                          const float *mlp_w, cudaStream_t st)
{
    k_spectrum<<<dim3((Kmax + 1 + 255) / 256, nsys), 256, 0, st>>>(spec, S);
    if (mlp_w) launch_spectrum_mlp(spec, nsys, Kmax, S, mlp_w, st);
    k_taps_table<<<dim3((Kmax + 1 + 127) / 128, nsys), 128, 0, st>>>(spec, S, cs);
    k_taps<<<dim3((Kmax + 1 + 31) / 32, nsys), 32, 0, st>>>(spec, S, cs, h64, h32);
}

void launch_kappa_solve(int P, int n, double ymax, double y0, double *A, double *b, double *M, double *r,
                        double *work, unsigned *err, cudaStream_t st)
{
    const int rows = 2 * n - 1, nt = (n + kCholNb - 1) / kCholNb, nmt = (rows + kCholNb - 1) / kCholNb, words = kappa_words(n);
    // scratch before the factorisation: the terms in M, the rows' scales and the tile flags in work
    // (small grids: too many terms for M, formed row by row)
    KappaTerm *terms = sizeof(KappaTerm) * (size_t)rows * P <= sizeof(double) * (size_t)n * n ? reinterpret_cast<KappaTerm *>(M) : nullptr;
    double *sc = work;
    // (nmt words <= 2 n ints up to n = 2^15; beyond, no tile is skipped)
    unsigned *nz = n <= (1 << 15) ? reinterpret_cast<unsigned *>(work + rows) : nullptr;
    cudaMemsetAsync(A, 0, sizeof(double) * (size_t)rows * n, st);
    if (terms) k_kappa_terms<<<dim3((rows + 127) / 128, P), 128, 0, st>>>(P, n, ymax, y0, terms);
    k_kappa_rows<<<(rows + 31) / 32, 32, 0, st>>>(P, n, ymax, y0, terms, A, b, sc);
    if (nz) cudaMemsetAsync(nz, 0, sizeof(unsigned) * (size_t)nmt * words, st);
    k_kappa_scale<<<nmt, 256, 0, st>>>(n, sc, A, nz, words);
    k_kappa_normal<<<nt * (nt + 1) / 2, 256, 0, st>>>(n, A, nz, words, M);
    if (nt > 1) k_kappa_envelope<<<nt, 64, 0, st>>>(n, nz, words, M);
    k_kappa_atv<<<nt, 256, 0, st>>>(n, A, b, r);
    chol_blocked(n, M, err, st);
    k_kappa_trsv<<<1, 32 * kTrsvWarps, 0, st>>>(n, M, r);
    double *s = work, *g = work + rows;
    for (int it = 0; it < kKappaRefine; ++it) {
        k_kappa_resid<<<(rows * 32 + 255) / 256, 256, 0, st>>>(rows, n, A, b, r, s);
        k_kappa_atv<<<nt, 256, 0, st>>>(n, A, s, g);
        k_kappa_trsv<<<1, 32 * kTrsvWarps, 0, st>>>(n, M, g);
        k_kappa_add<<<(n + 255) / 256, 256, 0, st>>>(n, r, g);
    }
}

size_t fourier_smem(int n, int fp64) { return (size_t)2 * kSegPairs * 2 * n * (fp64 ? 8 : 4); }

cudaError_t fourier_prepare(int n)
{
    const cudaError_t e = allow_dynamic_smem(k_fourier<float, float>, fourier_smem(n, 0));
    return e != cudaSuccess ? e : allow_dynamic_smem(k_fourier<double, double>, fourier_smem(n, 1));
}

void launch_spectrum_seg(const DSpec *spec, int nsys, int n, void *sq, int fp64, cudaStream_t st)
{
    dim3 g((unsigned)((n / 2 + 1 + 255) / 256), (unsigned)nsys);
    if (fp64) k_spectrum_seg<double><<<g, 256, 0, st>>>(spec, n, reinterpret_cast<double *>(sq));
    else k_spectrum_seg<float><<<g, 256, 0, st>>>(spec, n, reinterpret_cast<float *>(sq));
}

void launch_fourier(const Dev &d, int fp64, int max_dofp, int nsys, const void *sq, const void *tw, int n, int force,
                    cudaStream_t st)
{
    dim3 g((unsigned)((max_dofp + 2 * kSegPairs - 1) / (2 * kSegPairs)), (unsigned)nsys);
    const size_t sm = fourier_smem(n, fp64);
    if (fp64)
        k_fourier<double, double><<<g, 256, sm, st>>>(d, reinterpret_cast<const double *>(sq),
                                                      reinterpret_cast<const double *>(tw), n, force);
    else
        k_fourier<float, float><<<g, 256, sm, st>>>(d, reinterpret_cast<const float *>(sq),
                                                    reinterpret_cast<const float *>(tw), n, force);
}

}  // namespace qtb
