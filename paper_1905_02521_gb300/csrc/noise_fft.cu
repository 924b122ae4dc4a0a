// noise_fft.cu -- the FP64 coloured-noise filter (Eqs. 6-7) of long taps as a
// partitioned fast convolution in blocks of 256 steps.
//
// eta_n = sum_m g_m xi_{n + K_e - m}, g_m = h_|m - K_e|, K_e = 256 K_b.  Splitting g
// into parts g^q of 256 taps, block b of eta is the last half of a 512-point circular
// convolution,
//   eta_b = last 256 of IFFT( sum_q H_q (W_{b+K_b-q-1} + s W_{b+K_b-q}) ),
// H_q = FFT(g^q, 0), W_c = FFT(xi_c, 0) of one white block padded to 512 points and
// s_f = (-1)^f (a shift by half the length).  So a white block is transformed once,
// when it is drawn, and kept as its spectrum; with G_q = s H_q + H_{q-1} a block of
// noise is sum_{q=0}^{2 K_b} G_q W_{b+K_b-q} and one inverse transform.  (The term q =
// 2 K_b + 1 only reaches the discarded half: part 2 K_b has a single tap.)  Two dofs
// make one complex sequence: the taps are real, so real and imaginary part stay apart.
//
// The direct sum is bound by the FP64 pipes (2 K instructions a value; this GPU's FP64
// rate is 1/64 of its FP32 rate), this form does ~140 a value at 2049 taps: 5248 dofs,
// a block of noise in 0.35 ms (0.1 ms of it the drawing) instead of 4.9.
// The FP32 form keeps the direct sum (noise.cu): its rounding is part of trajectories
// that amplify any change of it beyond FP32 (double wells).
#include <cuda_runtime.h>

#include "qtb_dev.cuh"
#include "qtb_kernels.cuh"
#include "qtb_normal.cuh"

namespace qtb {

constexpr int kFftN = 2 * kBlockSteps;  // 512 points = 8 x 8 x 8
constexpr int kFftT = 64;               // threads of a transform, 8 points each

struct Cx {
    double x, y;
};
__device__ __forceinline__ Cx operator+(Cx a, Cx b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Cx operator-(Cx a, Cx b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Cx mul(Cx a, Cx b)
{
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// times S i (S = +1 inverse, -1 forward)
template <int S> __device__ __forceinline__ Cx muli(Cx a) { return S > 0 ? Cx{-a.y, a.x} : Cx{a.y, -a.x}; }

// 4- and 8-point transforms sum_k v_k e^{S 2 pi i k n/8}, natural order
template <int S> __device__ __forceinline__ void dft4(Cx &a, Cx &b, Cx &c, Cx &d)
{
    const Cx p = a + c, m = a - c, q = b + d, n = muli<S>(b - d);
    a = p + q; b = m + n; c = p - q; d = m - n;
}
template <int S> __device__ __forceinline__ void dft8(Cx (&v)[8])
{
    const double h = 0.70710678118654752440;
    Cx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<S>(e0, e1, e2, e3);
    dft4<S>(o0, o1, o2, o3);
    const Cx i1 = muli<S>(o1), i3 = muli<S>(o3);
    o1 = Cx{(o1.x + i1.x) * h, (o1.y + i1.y) * h};    // times e^{S i pi/4}
    o2 = muli<S>(o2);
    o3 = Cx{(i3.x - o3.x) * h, (i3.y - o3.y) * h};    // times e^{S 3 i pi/4}
    v[0] = e0 + o0; v[1] = e1 + o1; v[2] = e2 + o2; v[3] = e3 + o3;
    v[4] = e0 - o0; v[5] = e1 - o1; v[6] = e2 - o2; v[7] = e3 - o3;
}

// shared-memory exchange area of one transform (complex words); the row paddings
// keep every half-warp's 8-byte accesses on different banks
constexpr int kEx1 = 72, kEx2 = 66, kExSize = 8 * kEx1;

// twiddles of thread t: a[k] = e^{2 pi i t k/512}, b[k] = e^{2 pi i (t mod 8) k/64}
struct FftTw {
    Cx a[8], b[8];
    __device__ void load(const Cx *tw, int t)
    {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            a[k] = tw[(t * k) & (kFftN - 1)];
            b[k] = tw[(8 * (t & 7) * k) & (kFftN - 1)];
        }
    }
};

// 512-point transform over 64 threads: in v[k] = x[64 k + t], out v[c] = X[t + 64 c].
// Every thread of the CTA calls it (its barriers are the CTA's).
template <int S> __device__ __forceinline__ void fft512(Cx (&v)[8], const FftTw &tw, Cx *ex, int t)
{
    dft8<S>(v);
    __syncthreads();  // the exchange area is free
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const Cx w = S > 0 ? tw.a[k] : Cx{tw.a[k].x, -tw.a[k].y};
        ex[k * kEx1 + t] = k ? mul(v[k], w) : v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ex[(t >> 3) * kEx1 + (t & 7) + 8 * k];
    dft8<S>(v);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const Cx w = S > 0 ? tw.b[k] : Cx{tw.b[k].x, -tw.b[k].y};
        ex[(t & 7) * kEx2 + k * 8 + (t >> 3)] = k ? mul(v[k], w) : v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ex[k * kEx2 + t];
    dft8<S>(v);
}

// Draw white block blk (LLONG_MIN: clock + K_b) of every pair of dofs and store its
// spectrum: ring[slot][pair][512].  64 threads per pair, 4 pairs per CTA.
// grid = (max dofp / 8, nsys)
__global__ void __launch_bounds__(256) k_white_fft(Dev d, long long blk_override)
{
    __shared__ Cx ex_s[4][kExSize];
    const DSys s = d.sys[blockIdx.y];
    const int t = threadIdx.x & (kFftT - 1);
    const int dof = (blockIdx.x * 4 + threadIdx.x / kFftT) * 2;  // first dof of the pair, within the system
    if (blockIdx.x * 8 >= s.dofp || !s.fft) return;
    Cx *ex = ex_s[threadIdx.x / kFftT];
    FftTw tw;
    tw.load(reinterpret_cast<const Cx *>(d.fft_tw), t);
    const long long blk = (blk_override == LLONG_MIN) ? d.clock[0] + d.Kb : blk_override;
    const int slot = (int)(blk - floor_div(blk, d.nslots) * d.nslots);
    // one Philox call: 4 steps of one dof
#pragma unroll
    for (int ab = 0; ab < 2; ++ab) {
        double z[4] = {0, 0, 0, 0};
        if (dof + ab < 3 * s.N * s.P) white4(d, blockIdx.y, dof + ab, blk * (kBlockSteps / 4) + t, z);
#pragma unroll
        for (int q = 0; q < 4; ++q) (&ex[4 * t + q].x)[ab] = z[q];
    }
    __syncthreads();
    Cx v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k < 4 ? ex[64 * k + t] : Cx{0, 0};
    fft512<-1>(v, tw, ex, t);
    Cx *dst = reinterpret_cast<Cx *>(d.ring) + ((size_t)slot * (d.Dtot / 2) + (s.dof0 + dof) / 2) * kFftN;
#pragma unroll
    for (int c = 0; c < 8; ++c) dst[t + 64 * c] = v[c];
}

// eta of the current block.  A CTA takes kFftPairs pairs (their rows of eta: a full
// line), 4 at a time.  grid = (max dofp / (2 kFftPairs), nsys)
constexpr int kFftPairs = 8;
__global__ void __launch_bounds__(256, 2) k_filter_fft(Dev d)
{
    constexpr int NP = kFftPairs;
    extern __shared__ __align__(16) unsigned char fsm[];
    Cx *out = reinterpret_cast<Cx *>(fsm);                  // [256][NP + 1] outputs of the CTA's pairs
    Cx *ex = out + kBlockSteps * (NP + 1) + (threadIdx.x / kFftT) * kExSize;
    const DSys s = d.sys[blockIdx.y];
    const int t = threadIdx.x & (kFftT - 1);
    const int dof0 = blockIdx.x * 2 * NP;
    if (dof0 >= s.dofp || !s.fft) return;
    FftTw tw;
    tw.load(reinterpret_cast<const Cx *>(d.fft_tw), t);
    const long long b = d.clock[0];
    const Cx *G = reinterpret_cast<const Cx *>(d.fft_g) + (size_t)blockIdx.y * d.nslots * kFftN;
    for (int p0 = 0; p0 < NP; p0 += 4) {
        const int p = p0 + threadIdx.x / kFftT;
        const size_t pair = (size_t)(s.dof0 + dof0) / 2 + p;
        Cx v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = Cx{0, 0};
        for (int q = 0; q < d.nslots; ++q) {
            const long long c = b + d.Kb - q;
            const int slot = (int)(c - floor_div(c, d.nslots) * d.nslots);
            const Cx *w = reinterpret_cast<const Cx *>(d.ring) + ((size_t)slot * (d.Dtot / 2) + pair) * kFftN + t;
            const Cx *g = G + q * kFftN + t;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const Cx a = g[64 * k], x = w[64 * k];
                v[k].x = fma(a.x, x.x, fma(-a.y, x.y, v[k].x));
                v[k].y = fma(a.x, x.y, fma(a.y, x.x, v[k].y));
            }
        }
        fft512<1>(v, tw, ex, t);
#pragma unroll
        for (int c = 4; c < 8; ++c) out[(t + 64 * (c - 4)) * (NP + 1) + p] = v[c];
    }
    __syncthreads();
    double *eta = reinterpret_cast<double *>(d.eta);
    for (int e = threadIdx.x; e < kBlockSteps * 2 * NP; e += blockDim.x) {
        const int j = e / (2 * NP), l = e - j * 2 * NP;
        const Cx z = out[j * (NP + 1) + l / 2];
        eta[(size_t)j * d.Dtot + s.dof0 + dof0 + l] = (l & 1) ? z.y : z.x;
    }
}

// G_q of every system from its FP64 taps (the inverse transform's 1/512 included).
// grid = (nslots, nsys), 512 threads (one per frequency)
__global__ void __launch_bounds__(kFftN) k_fft_taps(Dev d, const double *taps, Cx *G)
{
    __shared__ double cs[kFftN], sn[kFftN], h[2][kBlockSteps];
    const DSys s = d.sys[blockIdx.y];
    if (!s.fft) return;
    const int q = blockIdx.x, f = threadIdx.x, Ke = kBlockSteps * d.Kb;
    sincospi(2.0 * f / kFftN, &sn[f], &cs[f]);
    for (int e = f; e < 2 * kBlockSteps; e += kFftN) {
        // part q - 1 (row 0) and q (row 1) of the taps
        const int m = (q - 1) * kBlockSteps + e, k = m - Ke, ka = k < 0 ? -k : k;
        h[e / kBlockSteps][e % kBlockSteps] = (m >= 0 && ka <= s.K) ? taps[s.taps0 + ka] : 0.0;
    }
    __syncthreads();
    double re = 0.0, im = 0.0;
    const double sg = (f & 1) ? -1.0 : 1.0;
    for (int r = 0; r < kBlockSteps; ++r) {
        const int a = (f * r) & (kFftN - 1);
        const double g = h[0][r] + sg * h[1][r];
        re = fma(g, cs[a], re);
        im = fma(-g, sn[a], im);
    }
    G[((size_t)blockIdx.y * d.nslots + q) * kFftN + f] = Cx{re / kFftN, im / kFftN};
}

__global__ void k_fft_twiddles(Cx *tw)
{
    double s, c;
    sincospi(2.0 * threadIdx.x / kFftN, &s, &c);
    tw[threadIdx.x] = Cx{c, s};
}

// ---------------------------------------------------------------------------
// launchers

constexpr size_t kFftSmem = sizeof(Cx) * (size_t)(kBlockSteps * (kFftPairs + 1) + 4 * kExSize);

size_t fft_table_values(int nslots, int nsys) { return 2 * (size_t)kFftN * ((size_t)nslots * nsys + 1); }

cudaError_t filter_fft_prepare()
{
    return allow_dynamic_smem(k_filter_fft, kFftSmem);
}

void launch_fft_tables(const Dev &d, const double *taps64, void *tw, void *G, cudaStream_t st)
{
    k_fft_twiddles<<<1, kFftN, 0, st>>>(reinterpret_cast<Cx *>(tw));
    k_fft_taps<<<dim3((unsigned)d.nslots, (unsigned)d.nsys), kFftN, 0, st>>>(d, taps64, reinterpret_cast<Cx *>(G));
}

void launch_white_fft(const Dev &d, int max_dofp, long long blk, cudaStream_t st)
{
    k_white_fft<<<dim3((unsigned)(max_dofp / 8), (unsigned)d.nsys), 256, 0, st>>>(d, blk);
}

void launch_filter_fft(const Dev &d, int max_dofp, cudaStream_t st)
{
    k_filter_fft<<<dim3((unsigned)(max_dofp / (2 * kFftPairs)), (unsigned)d.nsys), 256, kFftSmem, st>>>(d);
}

}  // namespace qtb
