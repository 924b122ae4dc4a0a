// ext.cu -- whole runs of steps of systems in a separable external potential, one
// launch for many steps (up to P = 8 beads; longer rings step by step, md.cu).
//
// Nothing couples the atoms of such a system, so a thread (or four, see ext_lanes)
// keeps one Cartesian component of one atom with all its beads in registers and carries
// it through the steps of the launch: B(dt/2), beads -> modes, A(dt/2) O(dt) A(dt/2), modes -> beads,
// force, B(dt/2).  The arithmetic is that of k_integrate(_nm) and k_force_ext, operation
// for operation (this file too is compiled without contraction), so a run gives the
// same bits however it is cut into launches.  What is left per step is the coloured
// noise, read once (fetched a step ahead, and a few more into the L2), instead of three
// launches that each stream the state.  Measured, 10923 atoms x 8 beads, mixed form,
// a record every 8 steps: 1.9 us a step instead of 32.
//
// Recorded steps: sums over a thread's beads in float-float (FP64 form: FP64), over
// the CTA in FP64, into a row per record and CTA; k_ext_records then forms the records.
#include "md_kernels.cuh"

namespace qtb {

constexpr int kExtAtoms = 32;                  // atoms of a CTA: warp c takes component c
constexpr int kExtThreads = 3 * kExtAtoms;
constexpr int kExtAhead = 6;                   // steps of noise prefetched into the L2
// row of a record: sums over the CTA's bead-atoms
enum { E_K = 0, E_V, E_X2, E_MOM, E_VIR = 6, E_SPRING = 9, E_CV, E_K0, E_N };
static_assert(E_N <= kExtRow, "row of a record");

// sum of products / values of the beads, error-free in the FP32 form
template <class R> struct Sum;
template <> struct Sum<float> {
    FF a{0.f, 0.f};
    __device__ void add(float v) { a.add(v); }
    __device__ void prod(float x, float y)
    {
        const float p = x * y;
        a.add_ff(p, fmaf(x, y, -p));
    }
    __device__ double value() const { return (double)a.hi + (double)a.lo; }
};
template <> struct Sum<double> {
    double s = 0.0;
    __device__ void add(double v) { s += v; }
    __device__ void prod(double x, double y) { s = fma(x, y, s); }
    __device__ double value() const { return s; }
};

// Sums of eight values over a warp by halving: each exchange leaves a lane with half of its
// values, so that the sums take 9 FP64 additions instead of the 40 of eight butterflies (a
// warp's FP64 instruction holds its quarter of the SM for 64 cycles).  2 million one-bead atoms,
// FP32 form, a record every step: 503 us a step, 815 with butterflies, 689 with a launch for
// every part of a step; FP64 form 1114, 1423, 1383.  Value q ends on lane 4 q.
__device__ __forceinline__ double warp_sum8(const double (&w)[8], int lane)
{
    double a[4], b[2];
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = (h16 ? w[4 + k] : w[k]) + __shfl_xor_sync(0xffffffffu, h16 ? w[k] : w[4 + k], 16);
#pragma unroll
    for (int k = 0; k < 2; ++k) b[k] = (h8 ? a[2 + k] : a[k]) + __shfl_xor_sync(0xffffffffu, h8 ? a[k] : a[2 + k], 8);
    double s = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

template <class R> __device__ __forceinline__ R ext_force(const PairTabT<R> &T, R kx, R x, R &e)
{
    if (T.potential == QTB_POT_HARMONIC) {
        e = R(0.5) * kx * x * x;
        return -kx * x;
    }
    const R u = x * x * T.ext_ia2 - R(1);
    e = T.ext_V0 * u * u;
    return R(-4) * T.ext_V0 * u * x * T.ext_ia2;
}

// L lanes share a component: its beads and modes are dealt to them, B = P / L each, and the
// transforms get the others' by shuffles, in the order one lane would take them.
template <int P, int L, class R>
__global__ void __launch_bounds__(kExtThreads * L) k_ext_steps(Dev d, PairTabT<R> T, int j0, int count)
{
    constexpr int B = P / L, A = 32 / L;  // A: atoms of a warp
    static_assert(P % L == 0 && (L == 1 || sizeof(R) == 8), "lanes of a component");
    __shared__ __align__(16) R Cs[P * P], CsT[P * P];
    __shared__ double red[3 * L][E_N];
    const int2 unit = d.ext_units[blockIdx.x];
    const DSys &S = d.sys[unit.x];
    if (S.P != P) return;  // another instantiation's (uniform over the CTA)
    for (int t = threadIdx.x; t < P * P; t += kExtThreads * L) {
        const R *Cg = reinterpret_cast<const R *>(d.nmC) + S.nm0;
        Cs[t] = Cg[t];                          // [b][k]
        CsT[t] = Cg[(t % P) * P + t / P];       // [k][b]
    }
    __syncthreads();
    const int N = S.N, warp = threadIdx.x >> 5, c = warp / L, lane = threadIdx.x & 31;
    const int la = lane % A, b0 = L == 1 ? 0 : lane / A * B;  // atom of the warp; first bead and mode of this lane
    const int i = unit.y + warp % L * A + la;
    const bool act = i < N;
    // value u of a component (u < P), held by one of its lanes in v[u % B]
    auto all = [&](const R (&v)[B], int u) { return L == 1 ? v[u % B] : __shfl_sync(0xffffffffu, v[u % B], u / B * A + la); };
    // sum of the component's lanes' values, in their order
    auto lanes_sum = [&](double v) {
        if constexpr (L == 1) return v;
        double s = __shfl_sync(0xffffffffu, v, la);
#pragma unroll
        for (int g = 1; g < L; ++g) s += __shfl_sync(0xffffffffu, v, g * A + la);
        return s;
    };
    const size_t G = (size_t)d.G, o = (size_t)c * G + S.g0 + (size_t)b0 * N + (act ? i : 0);
    R *X = reinterpret_cast<R *>(d.x), *V = reinterpret_cast<R *>(d.v), *F = reinterpret_cast<R *>(d.f);
    const int ty = d.typ[S.g0 + (act ? i : 0)];
    const R hdtm = T.hdt_m[ty], kx = T.ext_k[ty];
    const double m = T.mass[ty], hmv = 0.5 * T.mass_mvv[ty], w2 = S.wP * S.wP;
    const R sig = reinterpret_cast<const R *>(d.osig)[unit.x * kMaxTypes + ty];
    const R c1 = sizeof(R) == 4 ? (R)S.c1_f : (R)S.c1, invP = sizeof(R) == 4 ? (R)S.invP_f : (R)S.invP;
    R cs[B], sw[B], ws[B];
    {
        const R *rot = reinterpret_cast<const R *>(d.rot) + 3 * (S.rot0 + b0);
#pragma unroll
        for (int k = 0; k < B; ++k) {
            cs[k] = rot[3 * k]; sw[k] = rot[3 * k + 1]; ws[k] = rot[3 * k + 2];
        }
    }
    const R *eta = reinterpret_cast<const R *>(d.eta) + S.dof0 + (size_t)(3 * b0 + c) * N + (act ? i : 0);
    const size_t row0 = eta_row(d, 0);
    R x[B], v[B], f[B], en[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        x[b] = X[o + (size_t)b * N];
        v[b] = V[o + (size_t)b * N];
        f[b] = F[o + (size_t)b * N];
        en[b] = eta[(row0 + j0) * d.Dtot + (size_t)(3 * b) * N];
    }
    const long long base = d.clock[0] * kBlockSteps;
    const long long rec0 = (base + j0) / d.obs_stride;  // records before this launch
    for (int j = j0; j < j0 + count; ++j) {
        R nz[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            nz[k] = en[k];
            if (j + 1 < j0 + count) en[k] = eta[(row0 + j + 1) * d.Dtot + (size_t)(3 * k) * N];
            if (j + kExtAhead < j0 + count)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(eta + (row0 + j + kExtAhead) * d.Dtot + (size_t)(3 * k) * N));
        }
        // B(dt/2), beads relative to bead 0 -> modes
        R xr[B], q[B], p[B];
        const R xf = all(x, 0);
#pragma unroll
        for (int b = 0; b < B; ++b) {
            xr[b] = b0 + b == 0 ? R(0) : x[b] - xf;
            v[b] = fma(hdtm, f[b], v[b]);
            q[b] = p[b] = R(0);
        }
#pragma unroll
        for (int b = 0; b < P; ++b) {
            const R xb = all(xr, b), vb = all(v, b);
#pragma unroll
            for (int k = 0; k < B; ++k) {
                q[k] = fma(Cs[b * P + b0 + k], xb, q[k]);
                p[k] = fma(Cs[b * P + b0 + k], vb, p[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < B; ++k) mode_aoa(q[k], p[k], cs[k], sw[k], ws[k], c1, sig * nz[k]);
        R xn[B];
#pragma unroll
        for (int b = 0; b < B; ++b) xn[b] = v[b] = R(0);
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const R qk = all(q, k), pk = all(p, k);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                xn[b] = fma(CsT[k * P + b0 + b], qk, xn[b]);
                v[b] = fma(CsT[k * P + b0 + b], pk, v[b]);
            }
        }
        const long long step = base + j + 1;
        const bool rec = step % d.obs_stride == 0;
        Sum<R> sK, sV, sX, sM, sF, sS;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            x[b] = x[b] + (xn[b] - xr[b]);
            R e;
            const R fx = ext_force(T, kx, x[b], e);
            f[b] = fx * invP;
            v[b] = v[b] + hdtm * f[b];
            if (rec) {
                sK.prod(v[b], v[b]);
                sV.add(e);
                sX.prod(x[b], x[b]);
                sM.add(v[b]);
                sF.prod(x[b], fx);
            }
        }
        if (rec) {  // uniform
            double cv = 0.0, k0 = 0.0;
            if (P > 1) {
                Sum<R> sd, sv, sc;
                const R xe = L == 1 ? xn[0] : __shfl_sync(0xffffffffu, xn[0], (lane + A) & 31);  // the bead after the last
                const R x0 = all(x, 0);
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const R dx = xn[b] - (b + 1 < B ? xn[(b + 1) % B] : xe);
                    sS.add(dx * dx);
                    sd.add(x[b] - x0);
                    sv.add(v[b]);
                }
                const R dbar = (R)lanes_sum(sd.value()) * invP;
#pragma unroll
                for (int b = 0; b < B; ++b) sc.prod((x[b] - x0) - dbar, f[b]);
                const double vb = lanes_sum(sv.value()) * S.invP;
                cv = sc.value();
                k0 = b0 == 0 ? hmv * P * vb * vb : 0.0;
            }
            double w[8] = {hmv * sK.value(), sV.value(), sX.value(), m * sM.value(), sF.value(), cv, k0,
                           P > 1 ? hmv * w2 * sS.value() : 0.0};
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = act ? w[u] : 0.0;
            const double t = warp_sum8(w, lane);
            __syncthreads();  // the previous record's row is written
            if (lane < E_N) red[warp][lane] = 0.0;
            __syncwarp();
            if ((lane & 3) == 0) {
                const int u = lane >> 2;
                red[warp][u == 0 ? E_K : u == 1 ? E_V : u == 2 ? E_X2 : u == 3 ? E_MOM + c : u == 4 ? E_VIR + c
                          : u == 5 ? E_CV : u == 6 ? E_K0 : E_SPRING] = t;
            }
            __syncthreads();
            if (threadIdx.x < E_N) {
                double r = red[0][threadIdx.x];
#pragma unroll
                for (int u = 1; u < 3 * L; ++u) r += red[u][threadIdx.x];
                d.ext_part[((size_t)(step / d.obs_stride - 1 - rec0) * d.n_ext_units + blockIdx.x) * kExtRow + threadIdx.x] = r;
            }
        }
    }
    if (act) {
#pragma unroll
        for (int b = 0; b < B; ++b) {
            X[o + (size_t)b * N] = x[b];
            V[o + (size_t)b * N] = v[b];
            F[o + (size_t)b * N] = f[b];
        }
    }
}

// Records of a launch of k_ext_steps: record number rec0 + blockIdx.x of system
// blockIdx.y, summed over the system's CTAs in a fixed order (thread, then warp).
// grid = (most records of a launch, nsys), 128 threads
__global__ void __launch_bounds__(128) k_ext_records(Dev d, int j0, int count)
{
    __shared__ double sh[4][E_N], tot[E_N];
    const int s = blockIdx.y;
    const DSys &S = d.sys[s];
    if (S.P > kExtMaxP) return;
    const long long base = d.clock[0] * kBlockSteps, rec0 = (base + j0) / d.obs_stride;
    const long long rr = rec0 + blockIdx.x, step = (rr + 1) * d.obs_stride;
    if (step > base + j0 + count) return;
    double a[E_N];
#pragma unroll
    for (int u = 0; u < E_N; ++u) a[u] = 0.0;
    for (int e = S.eu0 + (int)threadIdx.x; e < S.eu1; e += blockDim.x)
#pragma unroll
        for (int u = 0; u < E_N; ++u) a[u] += d.ext_part[((size_t)blockIdx.x * d.n_ext_units + e) * kExtRow + u];
#pragma unroll
    for (int u = 0; u < E_N; ++u) {
        a[u] = warp_sum(a[u]);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][u] = a[u];
    }
    __syncthreads();
    if (threadIdx.x < E_N) tot[threadIdx.x] = (sh[0][threadIdx.x] + sh[1][threadIdx.x]) + (sh[2][threadIdx.x] + sh[3][threadIdx.x]);
    __syncthreads();
    const int q = threadIdx.x;
    if (q >= QTB_NREC) return;
    const double invP = S.invP, K = tot[E_K], V = tot[E_V] * invP, kT = 1.5 * S.N * kBoltz * S.T;
    const double vir[3] = {tot[E_VIR] * invP, tot[E_VIR + 1] * invP, tot[E_VIR + 2] * invP};
    const bool ring = S.P > 1;
    double r = 0.0;
    if (q == 0) r = (double)step;
    else if (q == 1) r = K;
    else if (q == 2) r = V;
    else if (q == 3) r = tot[E_SPRING];
    else if (q == 4) r = K - tot[E_SPRING] + V;
    else if (q == 5 || q == 9 || q == 13) r = vir[(q - 5) / 4];
    else if (q >= 14 && q < 17) r = tot[E_MOM + q - 14];
    else if (q == 17) r = tot[E_X2] * invP;
    else if (q == 18) r = ring ? kT - 0.5 * tot[E_CV] : kT;
    else if (q == 19) r = ring ? tot[E_K0] - 0.5 * tot[E_CV] : K;
    else if (q == 20) r = S.box[0] * S.box[1] * S.box[2];
    else if (q == 21) r = ring ? tot[E_K0] : K;
    else if (q == 22) r = (vir[0] + vir[1]) + vir[2] - (ring ? tot[E_CV] : 0.0);
    if (q == 0 && (!isfinite(K) || !isfinite(V))) atomicOr(d.err, (unsigned)ERR_NONFINITE);
    d.series[((size_t)(rr % d.max_records) * d.nsys + s) * QTB_NREC + q] = r;
    if (step + d.obs_stride > base + j0 + count) d.latest[(size_t)s * QTB_NREC + q] = r;
}

// lanes of a component: one, but four for rings of 8 beads in FP64, whose 400 FP64
// instructions a step are a chain of 16 us in one lane.  300 atoms, us a step, launch by
// launch / one lane / four: 15.8 / 16.7 / 13.2; a call of one step 38 / 46 / 36.
template <int P, class R> constexpr int ext_lanes = P == 8 && sizeof(R) == 8 ? 4 : 1;

template <class R>
static void ext_steps(const Dev &d, const MdLaunch &m, const PairTabT<R> &T, int j0, int count, cudaStream_t st)
{
    for (int u = 0; u < m.nP; ++u) {
        switch (m.Pvals[u]) {
#define QTB_P(PP) case PP: k_ext_steps<PP, ext_lanes<PP, R>, R><<<d.n_ext_units, kExtThreads * ext_lanes<PP, R>, 0, st>>>(d, T, j0, count); break;
            QTB_P(1) QTB_P(2) QTB_P(3) QTB_P(4) QTB_P(5) QTB_P(6) QTB_P(8)
#undef QTB_P
            default: break;
        }
    }
}

void launch_ext_steps(const Dev &d, const MdLaunch &m, const PairTabT<float> &Tf, const PairTabT<double> &Td, int j0,
                      int count, int max_rec, cudaStream_t st)
{
    if (m.mixed) ext_steps<float>(d, m, Tf, j0, count, st);
    else ext_steps<double>(d, m, Td, j0, count, st);
    if (max_rec > 0) k_ext_records<<<dim3((unsigned)max_rec, (unsigned)d.nsys), 128, 0, st>>>(d, j0, count);
}

}  // namespace qtb
