// Level update (Algorithm 1 lines 2-7): for each layer, merge the sampled histograms with the
// weights lambda_z = N_z^2 / sum N_z^2 and minimise
//     sum_j int_{l_j}^{l_{j+1}} (l_{j+1} - u)(u - l_j) dF~(u)
// (Section 3.2 of the paper, the minimisation that follows Eq. MQV).  The paper gives the objective
// only; the solver is exact coordinate minimisation: with neighbours a < c fixed, the optimal level
// l solves  F~(l) = F~(c) - int_a^c (u - a)/(c - a) dF~(u).  F~ is piecewise linear (uniform density
// inside a histogram bin), so F~, its first moment and its inverse are closed forms.
//
// Coordinate descent stops at a local minimum, and the objective has several when the density is not log-concave
// (a step density already has two), so the descent runs from two starts, the quantiles of the mass above bin 0 and the
// uniform grid, and the end point with the smaller objective is kept (the uniform start's only if it is smaller by
// more than one part in 10^9, so that rounding does not decide between two copies of the same minimum).
//
// One CTA per layer.  The fit is a chain of up to 200 dependent half sweeps (odd levels, then even ones; levels of one parity
// only depend on the other), so latency bounds it and the chain is what is kept short: one warp per start, both at once;
// a lane keeps its pairs of one even and one odd level in registers with F~ and the first moment at each, so a half
// sweep evaluates F~ once per level, not at both neighbours of every level, and takes neighbours by shuffles, without
// barriers; the bin of a value follows from its exponent and its first four mantissa bits; the inverse first looks at
// the bin it found the sweep before and at that bin's neighbours, and its bin serves F~ as well; divisions by a bin's
// density use reciprocals made once.  WGAN shapes, 4 bits, 8 samples: 876 us with a CTA-wide sweep per parity and start and
// two binary searches per neighbour, about 100 us now.
// All arithmetic is fp64 and this file is compiled without FMA contraction so that the sequence of roundings is the
// plain one: on histograms of few samples F~ has plateaus, and which end of one a level takes hangs on the last bit.
#include "lq_internal.cuh"

namespace lq {

constexpr int kBins = 385;            // bins 0..384 carry density; bin 385 (u = 1) never adds variance
constexpr int kFitThreads = 128;
constexpr int kMaxSweeps = 100;

struct FitSmem {
    double e[kBins + 1];
    double mass[kBins];
    double dens[kBins];               // mass / bin width, and its reciprocal (0 for an empty bin)
    double rdens[kBins];
    double F[kBins + 1];
    double M1[kBins + 1];
    double M2[kBins + 1];
    double l[2][kMaxLevels];          // the two starts' levels
    double term[2][kMaxLevels];
    double obj[2];
    double lambda[LQ_MAX_WORKERS];
    double wsum;
    float out[kMaxLevels];
    int ok;
};

__device__ __forceinline__ double bin_edge(int i)
{
    if (i <= 0) return 0.0;
    const int o = (i - 1) >> 4, m = (i - 1) & 15;
    return ldexp(1.0 + (double)m * 0.0625, o - 24);
}

// the bin of x in [0, 1]: the largest i <= 384 with e[i] <= x
__device__ __forceinline__ int bin_of(double x)
{
    const int t = (__double2hiint(x) >> 16) - ((1023 - 24) << 4);                // sixteenths of octaves above 2^-24
    return t < 0 ? 0 : min(t + 1, kBins - 1);
}

struct Cdf { double F, m1; };        // F~(x) and int_0^x u dF~(u)

// The two at x inside bin i (e its lower edge, d its density, F and m1 the sums at e).
__device__ __forceinline__ Cdf cdf_in_bin(double x, double e, double d, double F, double m1)
{
    const double part = (x - e) * d;
    return Cdf{F + part, m1 + part * ((e + x) * 0.5)};
}

__device__ __forceinline__ Cdf cdf(const FitSmem& s, double x, int& bin)
{
    const int i = bin = bin_of(x);
    return cdf_in_bin(x, s.e[i], s.dens[i], s.F[i], s.M1[i]);
}

// int_0^x u^2 dF~(u); inside a bin int_{e0}^{x} u^2 = (mass in [e0, x]) * (e0^2 + e0 x + x^2) / 3
__device__ __forceinline__ double second_moment(const FitSmem& s, double x)
{
    const int i = bin_of(x);
    const double part = (x - s.e[i]) * s.dens[i];
    return s.M2[i] + part * ((s.e[i] * s.e[i] + s.e[i] * x + x * x) / 3.0);
}

// x > y for non-negative x and any y that is a number: the patterns order like the values (a comparison on the integer
// pipe, a fraction of a fp64 comparison's latency)
__device__ __forceinline__ bool above(double x, double y) { return __double_as_longlong(x) > __double_as_longlong(y); }

// n / d, rounded correctly, from r = 1 / d rounded correctly: the rounded product n r, corrected once by its exact
// remainder (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990).  The
// reciprocals are made once per fit, so no division of the inverse is left on the chain.
__device__ __forceinline__ double quotient(double n, double d, double r)
{
    const double q = n * r;
    return fma(fma(-q, d, n), r, q);
}

// A level with F~ and the first moment at it, and its bin.
struct Level { double x; Cdf c; int bin; };

// The level at which F~ reaches y, between a and c: the bin is the first whose upper end exceeds y, looked for at the
// level's last bin and its neighbours first.
__device__ __forceinline__ void invert(const FitSmem& s, double y, double a, double c, Level& l)
{
    const int down = max(l.bin - 1, 0), up = min(l.bin + 1, kBins - 1);
    const double f0 = s.F[down], f1 = s.F[l.bin], f2 = s.F[l.bin + 1], f3 = s.F[up + 1];
    int lo = above(f1, y) ? down : (above(f2, y) ? l.bin : up);
    bool past = false;
    if ((above(f0, y) && down > 0) || !above(f3, y)) {
        int hi = kBins;
        lo = 0;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (above(s.F[mid + 1], y)) hi = mid; else lo = mid + 1;
        }
        past = lo >= kBins;
        lo = min(lo, kBins - 1);
    }
    const double e = s.e[lo], F = s.F[lo], d = s.dens[lo], m1 = s.M1[lo];
    double w = quotient(y - F, d, s.rdens[lo]);
    if (__double2hiint(w) < 0) w = 0.0;
    double b = past ? 1.0 : e + w;
    if (above(a, b)) b = a;
    if (above(b, c)) b = c;
    l.x = b;
    l.bin = bin_of(b);
    l.c = cdf_in_bin(b, e, d, F, m1);
    if (l.bin != lo) l.c = cdf(s, b, l.bin);
}

// The exact minimiser between fixed neighbours a and c; true if it moved the level by more than 1e-13 of itself.
__device__ __forceinline__ bool relax(const FitSmem& s, Level& l, double a, const Cdf& ca, double c, const Cdf& cc)
{
    if (!above(c, a)) return false;
    const double mass_ac = cc.F - ca.F, before = l.x;
    if (!above(cc.F, ca.F)) {
        l.x = (a + c) * 0.5;
        l.c = cdf(s, l.x, l.bin);
    } else {
        invert(s, cc.F - ((cc.m1 - ca.m1) - a * mass_ac) / (c - a), a, c, l);
    }
    // |b - l| / max(|b|, 1e-300) > 1e-13: 450 to 901 units in the last place; divided out only where their number does not tell
    const long long ulps = llabs(__double_as_longlong(l.x) - __double_as_longlong(before));
    return ulps > 1000 || (ulps > 400 && fabs(l.x - before) / fmax(fabs(l.x), 1e-300) > 1e-13);
}

__device__ __forceinline__ Cdf shfl_cdf(const Cdf& c, int src)
{
    return Cdf{__shfl_sync(0xffffffffu, c.F, src), __shfl_sync(0xffffffffu, c.m1, src)};
}

// Odd/even sweeps of exact coordinate minimisation on the levels l (shared memory, n = 2^b of them), by one warp: lane t
// holds the pairs (2 q, 2 q + 1), q = V t .. V t + V - 1.
template <int V>
__device__ void descend(const FitSmem& s, double* l, int n, int lane)
{
    Level ev[V], od[V];
    const int pairs = n >> 1;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int q = V * lane + v;
        ev[v].x = q < pairs ? l[2 * q] : 1.0;
        od[v].x = q < pairs ? l[2 * q + 1] : 1.0;
        ev[v].c = cdf(s, ev[v].x, ev[v].bin);
        od[v].c = cdf(s, od[v].x, od[v].bin);
    }
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        bool moved = false;
        // odd levels: between this pair's even level and the next pair's
        {
            const double nx = __shfl_down_sync(0xffffffffu, ev[0].x, 1);
            const Cdf nc = shfl_cdf(ev[0].c, lane + 1);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const double c = v + 1 < V ? ev[(v + 1) % V].x : nx;
                const Cdf cc = v + 1 < V ? ev[(v + 1) % V].c : nc;
                if (V * lane + v < pairs - 1) moved |= relax(s, od[v], ev[v].x, ev[v].c, c, cc);
            }
        }
        // even levels: between the previous pair's odd level and this pair's
        {
            const double px = __shfl_up_sync(0xffffffffu, od[V - 1].x, 1);
            const Cdf pc = shfl_cdf(od[V - 1].c, lane - 1);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const double a = v > 0 ? od[(v + V - 1) % V].x : px;
                const Cdf ca = v > 0 ? od[(v + V - 1) % V].c : pc;
                const int q = V * lane + v;
                if (q >= 1 && q < pairs) moved |= relax(s, ev[v], a, ca, od[v].x, od[v].c);
            }
        }
        if (!__any_sync(0xffffffffu, moved)) break;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int q = V * lane + v;
        if (q < pairs) { l[2 * q] = ev[v].x; l[2 * q + 1] = od[v].x; }
    }
    __syncwarp();
}

// The objective at the levels l: interval j gives -(M2(c) - M2(a)) + (a + c)(M1(c) - M1(a)) - a c (F(c) - F(a));
// the intervals are added in order by one lane so that the sum does not depend on how they were dealt out.
__device__ void objective(const FitSmem& s, const double* l, int n, int lane, double* term, double* out)
{
    for (int j = lane; j + 1 < n; j += 32) {
        const double a = l[j], c = l[j + 1];
        int bin;
        const Cdf ca = cdf(s, a, bin), cc = cdf(s, c, bin);
        const double m2a = second_moment(s, a), m2c = second_moment(s, c);
        term[j] = ((a + c) * (cc.m1 - ca.m1) - (m2c - m2a)) - (a * c) * (cc.F - ca.F);
    }
    __syncwarp();
    if (lane == 0) {
        double total = 0.0;
        for (int j = 0; j + 1 < n; ++j) total += term[j];
        *out = total;
    }
}

// Per-layer mode (member_off == nullptr): CTA m fits layer m.  Shared mode: CTA t fits one sequence for type t,
// whose member layers are member_layer[member_off[t] .. member_off[t+1]) (all with the same level count): the
// histograms of all (sample, member) pairs are merged with weights N^2 (the variance to minimise is
// sum N_s^2 sum_i sigma^2(u_i)), scaled by sum N_s^2 d_s, and the result goes to every member.
__global__ void __launch_bounds__(kFitThreads) fit_levels_kernel(PlanDev p, const uint32_t* hist,
                                                                 const float* norms, int Z,
                                                                 float* levels_stage,
                                                                 const int32_t* member_off,
                                                                 const int32_t* member_layer)
{
    __shared__ FitSmem s;
    pdl_launch_next();
    pdl_wait();
    const bool shared_fit = member_off != nullptr;
    const int m0 = shared_fit ? member_off[blockIdx.x] : 0, m1 = shared_fit ? member_off[blockIdx.x + 1] : 0;
    if (shared_fit && m1 <= m0) return;
    const int m = shared_fit ? member_layer[m0] : blockIdx.x;
    const LayerDesc L = p.layers[m];
    const int n = L.nlevels;
    if (n < 3) return;
    const int tid = threadIdx.x;

    if (shared_fit) {
        if (tid == 0) {
            double wd = 0.0;
            for (int z = 0; z < Z; ++z)
                for (int j = m0; j < m1; ++j) {
                    const int mm = member_layer[j];
                    const double w = (double)norms[(int64_t)z * p.num_layers + mm];
                    wd += w * w * (double)p.layers[mm].size;
                }
            s.wsum = wd;
            s.ok = wd > 0.0;
        }
        __syncthreads();
        if (!s.ok) return;
        const double wd = s.wsum;
        for (int i = tid; i <= kBins; i += kFitThreads) s.e[i] = bin_edge(i);
        for (int i = tid; i < kBins; i += kFitThreads) {
            double acc = 0.0;
            for (int z = 0; z < Z; ++z)
                for (int j = m0; j < m1; ++j) {
                    const int mm = member_layer[j];
                    const double w = (double)norms[(int64_t)z * p.num_layers + mm];
                    acc += (w * w) * (double)hist[((int64_t)z * p.num_layers + mm) * LQ_HIST_STRIDE + i];
                }
            s.mass[i] = acc / wd;
        }
        __syncthreads();
    } else {
    if (L.size <= 0) return;

    for (int z = tid; z < Z; z += kFitThreads) {
        const double w = (double)norms[(int64_t)z * p.num_layers + m];
        s.lambda[z] = w * w;
    }
    __syncthreads();
    if (tid == 0) {
        double wsum = 0.0;
        for (int z = 0; z < Z; ++z) wsum += s.lambda[z];
        s.wsum = wsum;
        s.ok = wsum > 0.0;
    }
    __syncthreads();
    if (!s.ok) return;
    for (int z = tid; z < Z; z += kFitThreads) s.lambda[z] = s.lambda[z] / s.wsum;
    __syncthreads();

    for (int i = tid; i <= kBins; i += kFitThreads) s.e[i] = bin_edge(i);
    for (int i = tid; i < kBins; i += kFitThreads) {
        double acc = 0.0;
        for (int z = 0; z < Z; ++z)
            acc += s.lambda[z] * (double)hist[((int64_t)z * p.num_layers + m) * LQ_HIST_STRIDE + i];
        s.mass[i] = acc / (double)L.size;
    }
    __syncthreads();
    }
    // running sums of the mass and its first two moments: the terms by everybody, each chain of additions by one thread
    for (int i = tid; i < kBins; i += kFitThreads) {
        s.F[i + 1] = s.mass[i];
        s.M1[i + 1] = s.mass[i] * ((s.e[i] + s.e[i + 1]) * 0.5);
        s.M2[i + 1] = s.mass[i] * ((s.e[i] * s.e[i] + s.e[i] * s.e[i + 1] + s.e[i + 1] * s.e[i + 1]) / 3.0);
        s.dens[i] = s.mass[i] / (s.e[i + 1] - s.e[i]);         // (exact: a bin's width is a power of two)
        s.rdens[i] = s.mass[i] > 0.0 ? 1.0 / s.dens[i] : 0.0;
    }
    __syncthreads();
    if ((tid & 31) == 0 && tid < 96) {
        double* a = tid == 0 ? s.F : (tid == 32 ? s.M1 : s.M2);
        double run = 0.0;
        a[0] = run;
        constexpr int kAhead = 11;
        static_assert(kBins % kAhead == 0, "terms are fetched in whole groups");
        for (int i = 0; i < kBins; i += kAhead) {
            double t[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k) t[k] = a[1 + i + k];
#pragma unroll
            for (int k = 0; k < kAhead; ++k) { run += t[k]; a[1 + i + k] = run; }
        }
    }
    __syncthreads();
    const double mass_above = s.F[kBins] - s.mass[0];
    if (!(mass_above > 0.0)) return;

    for (int j = tid; j < n; j += kFitThreads) {
        const double frac = (double)j / (double)(n - 1);
        Level l{0.0, Cdf{0.0, 0.0}, kBins / 2};
        invert(s, s.mass[0] + mass_above * frac, 0.0, 1.0, l);
        s.l[0][j] = j == 0 || j == n - 1 ? frac : l.x;
        s.l[1][j] = frac;
    }
    __syncthreads();

    const int warp = tid >> 5, lane = tid & 31;
    if (warp < 2) {
        if (n <= 64)       descend<1>(s, s.l[warp], n, lane);
        else if (n <= 128) descend<2>(s, s.l[warp], n, lane);
        else               descend<4>(s, s.l[warp], n, lane);
        objective(s, s.l[warp], n, lane, s.term[warp], &s.obj[warp]);
    }
    __syncthreads();

    // round to fp32; force strict monotonicity (one ulp and 2^-40 above the level before, one ulp
    // below the level after; serial: order matters)
    if (tid == 0) {
        const double* l = s.l[s.obj[1] < s.obj[0] * (1.0 - 1e-9) ? 1 : 0];
        float before = 0.0f;
        s.out[0] = 0.0f; s.out[n - 1] = 1.0f;
        for (int j = 1; j <= n - 2; ++j) {
            const float f = (float)l[j];
            float fl = __uint_as_float(__float_as_uint(before) + 1u);               // the next float upwards
            const float gap = __fadd_rn(before, 9.094947017729282e-13f);           // previous level + 2^-40
            if (gap > fl) fl = gap;
            before = f > fl ? f : fl;
            s.out[j] = before;
        }
        float after = 1.0f;
        for (int j = n - 2; j >= 1; --j) {
            const float ce = __uint_as_float(__float_as_uint(after) - 1u);          // the next float downwards
            if (s.out[j] > ce) s.out[j] = ce;
            after = s.out[j];
        }
    }
    __syncthreads();
    for (int jm = m0; jm < m1 || jm == m0; ++jm) {         // in shared mode every member of the type receives the sequence
        float* dst = levels_stage + (int64_t)(shared_fit ? member_layer[jm] : m) * kLevelStride;
        for (int j = tid; j < n; j += kFitThreads) dst[j] = s.out[j];
    }
}

cudaError_t launch_fit(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                       float* levels_stage, cudaStream_t s)
{
    if (p.num_layers == 0) return cudaSuccess;
    return launch(fit_levels_kernel, (unsigned)p.num_layers, kFitThreads, 0, s, p, hist, norms, num_samples, levels_stage,
                  nullptr, nullptr);
}

cudaError_t launch_fit_shared(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                              float* levels_stage, const int32_t* member_off, const int32_t* member_layer,
                              int num_types, cudaStream_t s)
{
    if (num_types == 0) return cudaSuccess;
    return launch(fit_levels_kernel, (unsigned)num_types, kFitThreads, 0, s, p, hist, norms, num_samples, levels_stage,
                  member_off, member_layer);
}

}  // namespace lq
