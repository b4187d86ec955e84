// Linear subdomain marches in 64-bit fixed point (arithmetic: swr_fx.cuh): constant matrices,
// and V(t,x) with every step's factors streamed.
//
// The march and its partition into chunks and separators are those of swr_march.cu
// (k_march_static, k_march_tl); the arithmetic is 5-6 times cheaper, which moves the limits:
//   * instruction fetch.  Straight-line code runs at 0.75 instructions per cycle and SM
//     sub-partition up to 12 KB, about 0.6 up to 40 KB and 0.25 beyond 56 KB (measured).  The
//     first form of this kernel (the chunk solve and spike correction of k_march_static, 360
//     instructions per node, 76 KB) spent 2.7 of 7 stall cycles on fetches: 8.6 ms for the
//     N = 500 build of the scaling workload.  The chunk work is therefore written with as
//     few instructions as the recurrences allow and the separator solve as loops;
//   * all right-hand sides of one subdomain (zero-flux march, left and right impulse) share a
//     CTA (or cluster) and its copy of the factors in shared memory, loaded once for all steps;
//   * a system of at most 32 separators is one warp and marches without any barrier; a
//     longer one takes one barrier per step (every warp solves the reduced system itself);
//   * end traces and recorded states leave as integers (an integer -> FP64 conversion costs
//     as much as a DFMA): k_fx_flux forms the fluxes of all steps afterwards and the
//     superposition reads integer states.
//
// A step of a chunk (T its matrix, f its right-hand side, vL and vR the separators' values):
//   forward   z_i = f_i - c_{i-1} z_{i-1},  and  sum_i a_i f_i = E_left (T^{-1} f)_first,
//             because T is symmetric and a = T^{-1} E_left e_first is the left spike;
//             c_last z_last = E_right (T^{-1} f)_last with c_last = q_last E_right;
//   separators from these two numbers per chunk;
//   backward  x_i = q_i z_i - g_i vL - c_i x_{i+1},  x_{L+1} = vR,  g_i = q_i za_i (za the
//             left coupling carried through the elimination), u_i <- 2 x_i - u_i.
// Five complex multiply-adds per node as in the two-sweep form, but two roundings instead of
// three.  A chunk with fewer than L nodes has its first slots filled with copies of its left
// separator (q = c = 0, g = -1: x = vL exactly), so the code has no conditions per node.
//
// Range.  The states of a system are scaled so that the largest component after step 1 is in
// [2^56, 2^57) ([2^55, 2^56) for a march with flux inputs).  With every |u| <= 2^58 the bounds
// computed with the factors (fx_sub) keep every intermediate of the next step within the
// limits of swr_fx.cuh, so a march whose checks pass has not wrapped anywhere: every
// component of every step is tested against a trigger, 2^57 (2^56); beyond it the system is
// scaled down by 4, and beyond 2^58 it is flagged.  Flagged systems (growth too fast for the
// trigger, non-finite data, factors outside the bounds, traces too small to keep enough bits,
// see k_fx_flux) are marched again in FP64 by the kernels of swr_march.cu.  The first step,
// which sets the scale, is always an FP64 one.
//
// Measured, build marches of 200001 nodes and 500 steps (zero flux, left and right impulse; first
// step, scales, march and fluxes), FP64 -> here: 500 subdomains 16.6 -> 4.7 ms, 256 19.4 -> 6.3, 64
// 18.9 -> 6.3, 16 19.5 -> 10.3 (bound by issue, about 240 instructions per node and step at 500; by
// a step's dependent chain and its separators' exchange at 16).  S_0^2 ends, 100003 nodes in 61
// subdomains, 300 steps: 7.5 -> 4.1.  1001 nodes in 4 subdomains, 200 steps, whole products: 1.65
// -> 1.01.  V(t,x), 60001 nodes in 64 subdomains, 400 steps: 4.76 -> 2.26 ms a march (one CTA of
// six warps per subdomain: the chain of a step, 5.6 us).
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "swr_fx.cuh"
#include "swr_internal.cuh"

namespace cg = cooperative_groups;

// ---------------------------------------------------------------------------
// Factors: range analysis (k_fx_bounds) and conversion (k_fx_convert).
//
// Scales (powers of two, per subdomain): z is formed at 2^-s of the state's scale, the
// separators' right-hand sides at 2^-s2, the separator solve runs at 2^-sd, the reduced one
// at 2^-sr.
// Moduli are bounded for states of unit components through the same recurrences in absolute
// values; the state limit 2^58 leaves a factor of 4 below 2^60.
// ---------------------------------------------------------------------------
namespace {
enum { B_Q, B_CO, B_GC, B_Z, B_Y, B_D, B_CZ, B_BI, B_AX, B_RI, B_CL, B_PG, B_RG = B_PG + 5, B_N = B_RG + 5 };
constexpr double kFxF = 8.5;   // |f| <= 6 sqrt(2) for unit components
// The absolute recurrences overestimate the separators' right-hand sides a little (smooth states
// come within a factor of two): their scales are finer by this many bits than the bounds allow,
// and every level's values are tested against 2^60 instead.
constexpr int kFxSlack = 1;
}

size_t swr_fx_bounds_bytes(int N) { return sizeof(unsigned long long) * B_N * (size_t)N; }

// |a| from above, at most 8 % over: sqrt(m^2 + n^2) <= m + (sqrt(2) - 1) n for n <= m (a square
// root is some twenty FP64 instructions)
__device__ __forceinline__ double cabs_(double2 a) {
    const double x = fabs(a.x), y = fabs(a.y);
    return x > y ? fma(0.41422, y, x) : fma(0.41422, x, y);
}

// maxima of subdomain j's coefficients and absolute recurrences into mx[j]; threads over
// chunks / separators p of one tile
__global__ void __launch_bounds__(64) k_fx_bounds(
    int L, int P, int levels, int one, const int* __restrict__ sub_P,
    const unsigned char* __restrict__ clen, const double2* __restrict__ fac,
    const double2* __restrict__ sep, const double2* __restrict__ pcr,
    const double2* __restrict__ tl_pcr, const double2* __restrict__ tl_aux,
    const double2* __restrict__ tl_red, unsigned long long* __restrict__ mx, long long fstride,
    long long sstride, long long pstride) {
    __shared__ unsigned long long sm[B_N];
    const int j = blockIdx.y, S = P + 1, p = blockIdx.x * blockDim.x + threadIdx.x;
    const int Pj = sub_P[j], Q = (Pj + 31) / 32, N = gridDim.y;
    {   // batch entry z (per-step factors)
        const size_t z = blockIdx.z;
        fac += z * fstride;
        sep += z * sstride;
        pcr += z * pstride;
        tl_pcr += z * N * 10 * S;
        tl_aux += z * N * 3 * S;
        tl_red += z * N * 13 * 32;
        mx += z * N * B_N;
    }
    for (int k = threadIdx.x; k < B_N; k += blockDim.x) sm[k] = 0;
    __syncthreads();
    // |x| of a finite or NaN double orders as an integer (NaN above everything)
    auto put = [&](int k, double v) {
        atomicMax(&sm[k], (unsigned long long)__double_as_longlong(fabs(v)));
    };
    const double2* E = sep + (size_t)j * 3 * S;
    if (p < Pj) {
        const double2* F = fac + (size_t)j * L * 4 * P + p;
        const int Lp = clen[j * P + p];
        const double El = cabs_(E[p + 1]);
        double z = 0, za = cabs_(E[S + p]), cp = 0, zm = 0, d = 0;
        for (int i = 0; i < Lp; ++i) {
            const double q = cabs_(F[(i * 4 + 0) * P]);
            const double c = i == Lp - 1 ? q * El : cabs_(F[(i * 4 + 1) * P]);
            const double a = cabs_(F[(i * 4 + 2) * P]);
            z = kFxF + cp * z;
            if (i) za *= cp;
            zm = zm > z ? zm : z;
            d += kFxF * a;
            put(B_CO, fmax(c, a));
            put(B_GC, c + q * za);
            put(B_Q, q);
            cp = c;
        }
        put(B_Z, zm);
        put(B_D, d);
        put(B_CZ, cp * z);
        double y = 0, ym = 0;
        for (int i = Lp - 1; i >= 0; --i) {
            y = cabs_(F[(i * 4 + 0) * P]) * zm + cabs_(F[(i * 4 + 1) * P]) * y;
            ym = fmax(ym, y);
        }
        put(B_Y, ym);
    }
    if (p <= Pj) {
        if (one) {
            put(B_BI, cabs_(E[2 * S + p]));
            for (int k = 0; k < levels && k < 5; ++k)
                put(B_PG + k, cabs_(pcr[((size_t)(j * levels + k) * 2 + 0) * S + p]) +
                                  cabs_(pcr[((size_t)(j * levels + k) * 2 + 1) * S + p]));
        } else {
            const double2* A = tl_aux + (size_t)j * 3 * S + p;
            const bool member = (p & 31) != 0 && p != Pj;
            if (member) put(B_BI, cabs_(A[0]));
            put(B_AX, cabs_(A[S]) + cabs_(A[2 * S]));
            for (int k = 0; k < 5; ++k)
                put(B_PG + k, cabs_(tl_pcr[((size_t)j * 10 + 2 * k) * S + p]) +
                                  cabs_(tl_pcr[((size_t)j * 10 + 2 * k + 1) * S + p]));
        }
    }
    if (!one && blockIdx.x == 0 && threadIdx.x <= Q && threadIdx.x < 32) {
        const double2* R = tl_red + (size_t)j * 13 * 32 + threadIdx.x;
        put(B_RI, cabs_(R[10 * 32]));
        put(B_CL, cabs_(R[11 * 32]) + cabs_(R[12 * 32]));
        for (int k = 0; k < 5; ++k) put(B_RG + k, cabs_(R[2 * k * 32]) + cabs_(R[(2 * k + 1) * 32]));
    }
    __syncthreads();
    for (int k = threadIdx.x; k < B_N; k += blockDim.x)
        if (sm[k]) atomicMax(&mx[(size_t)j * B_N + k], sm[k]);
}

// Scales of one subdomain from its maxima; eb, er, eC: exponents of 1/delta of the separators
// and of the reduced system, and of its couplings.
__device__ __forceinline__ FxSub fx_sub(const unsigned long long* mx, double hist, int& eb, int& er,
                                        int& eC) {
    auto get = [&](int k) { return __longlong_as_double((long long)mx[k]); };
    const double tiny = 1e-9;
    FxSub f = {};
    eb = er = eC = 0;
    bool bad = false;
    for (int k = 0; k < B_N; ++k) bad |= !isfinite(get(k)) || get(k) > 1e12;
    if (!bad) {
        double g1 = 1.0, g2 = 1.0;
        for (int k = 0; k < 5; ++k) {
            g1 *= 1.0 + get(B_PG + k);
            g2 *= 1.0 + get(B_RG + k);
            bad |= get(B_PG + k) > 2.6 || get(B_RG + k) > 2.6;
        }
        // x of the backward sweep: B_Y from the right-hand sides, and from vL and vR at most 1.42
        // for any grid (V = 0; 2.5 taken), 8 in all, |x| < 2^61.  B_Y overestimates by up to a
        // quarter: 4.25 at most for exact moduli, up to 5.3 from the recurrences of k_fx_bounds,
        // where dt/h^2 is about 0.2 or, with 12 nodes and more, 3 to 10.  (The limit was 4: all
        // marches of such a grid ran in FP64 in an untuned shape, a solve of 1355 nodes and 372
        // steps in 12.7 ms instead of 5.2.)
        bad |= get(B_CO) > 1.1 || get(B_AX) > 2.6 || get(B_Y) > 5.5;
        // a separator's row: its stencil and a flux, the two chunks' parts
        // (and with S_0^2 ends a history term of a few times |c2 / (i kappa)| v, tested as it comes)
        const double d0 = 2.0 * kFxF + get(B_D) + get(B_CZ) + 6.0 * hist;
        f.s = max(0, fx_clog2(fmax(get(B_Z), 1.0)) - 2);
        f.s2 = max(f.s, fx_clog2(fmax(d0, 1.0)) - 2);
        const double q = get(B_Q) * scalbn(1.0, f.s);
        bad |= f.s2 > 28 || q > 1.99 || q + get(B_GC) > 2.6;
        f.sd = max(f.s2, fx_clog2(fmax(d0 * g1, 1.0)) - 2 - kFxSlack);
        eb = -fx_clog2(fmax(get(B_BI), tiny));
        f.kv = eb - f.sd;
        // super-chunk values are checked against 2^58
        const double r0 = d0 + 1.5 * get(B_CL);
        eC = fx_clog2(fmax(get(B_CL), tiny));
        f.sr = max(f.s2, fx_clog2(fmax(r0 * g2, 1.0)) - 2 - kFxSlack);
        f.kc = f.sr - eC;
        er = -fx_clog2(fmax(get(B_RI), tiny));
        f.kr = er - f.sr;
        bad |= f.sd > 50 || f.sr > 50 || f.kv > 55 || f.kr > 55 || f.kv < -20 || f.kr < -20 ||
               f.kc > 60 || f.kc < -20;
    }
    f.bad = bad ? 1 : 0;
    return f;
}

// Rows of coefficients: [N][P+1][4 L + 13], per separator p
//   4 i + (0..3)     chunk slot i: q 2^s, -c, -a 2^-s2, -g
//   4 L + 2 k, + 1   PCR level k (of the system, or of its super-chunk)
//   4 L + 10         1 / delta 2^eb
//   4 L + 11, + 12   super-chunk spikes -a, -b
// and the reduced system [N][13][32].
__global__ void __launch_bounds__(64) k_fx_convert(
    int L, int P, int levels, int one, const int* __restrict__ sub_P,
    const unsigned char* __restrict__ clen, const double2* __restrict__ fac,
    const double2* __restrict__ sep, const double2* __restrict__ pcr,
    const double2* __restrict__ tl_pcr, const double2* __restrict__ tl_aux,
    const double2* __restrict__ tl_red, const unsigned long long* __restrict__ mx,
    FxSub* __restrict__ fsub, int4* __restrict__ rows, int4* __restrict__ red, long long fstride,
    long long sstride, long long pstride, double hist) {
    const int j = blockIdx.y, S = P + 1, p = blockIdx.x * blockDim.x + threadIdx.x;
    const int Pj = sub_P[j], Q = (Pj + 31) / 32, N = gridDim.y;
    {   // batch entry z (per-step factors)
        const size_t z = blockIdx.z;
        fac += z * fstride;
        sep += z * sstride;
        pcr += z * pstride;
        tl_pcr += z * N * 10 * S;
        tl_aux += z * N * 3 * S;
        tl_red += z * N * 13 * 32;
        mx += z * N * B_N;
        fsub += z * N;
        rows += z * N * S * (4 * L + 13);
        red += z * N * 13 * 32;
    }
    int eb, er, eC;
    const FxSub f = fx_sub(mx + (size_t)j * B_N, hist, eb, er, eC);
    if (blockIdx.x == 0 && threadIdx.x == 0) fsub[j] = f;
    if (f.bad) return;
    const double2 zero = make_double2(0.0, 0.0);
    auto coef = [&](double2 v, double sc) { return fx_coef(v.x * sc, v.y * sc); };
    const int4 nil = make_int4(0, 0, 0, 0);
    if (p < S) {
        int4* o = rows + ((size_t)j * S + p) * (4 * L + 13);
        const double2* E = sep + (size_t)j * 3 * S;
        const double2* F = fac + (size_t)j * L * 4 * P + (p < P ? p : 0);
        const int Lp = p < Pj ? clen[j * P + p] : 0, nv = L - Lp;
        const double qs = scalbn(1.0, f.s), as = -scalbn(1.0, -f.s2);
        double2 za = p < Pj ? E[S + p] : zero, cp = zero;
        for (int i = 0; i < L; ++i, o += 4) {
            if (i < nv) {   // a copy of the left separator
                o[0] = o[1] = o[2] = nil;
                o[3] = fx_coef(p <= Pj ? 1.0 : 0.0, 0.0);
                continue;
            }
            const int k = i - nv;
            const double2 q = F[(k * 4 + 0) * P];
            if (k) za = cmul(make_double2(-cp.x, -cp.y), za);
            cp = k == Lp - 1 ? cmul(q, E[p + 1]) : F[(k * 4 + 1) * P];
            o[0] = coef(q, qs);
            o[1] = coef(cp, -1.0);
            o[2] = coef(F[(k * 4 + 2) * P], as);
            o[3] = coef(cmul(q, za), -1.0);
        }
        const bool member = (p & 31) != 0 && p < Pj;
        const double2* A = tl_aux + (size_t)j * 3 * S + p;
        for (int k = 0; k < 10; ++k) {
            if (one)
                o[k] = coef(p <= Pj && (k >> 1) < levels
                                ? pcr[((size_t)(j * levels + (k >> 1)) * 2 + (k & 1)) * S + p] : zero, 1.0);
            else
                o[k] = coef(member ? tl_pcr[((size_t)j * 10 + k) * S + p] : zero, 1.0);
        }
        o[10] = coef(one ? (p <= Pj ? E[2 * S + p] : zero) : (member ? A[0] : zero), scalbn(1.0, eb));
        o[11] = coef(!one && member ? A[S] : zero, -1.0);
        o[12] = coef(!one && member ? A[2 * S] : zero, -1.0);
    }
    if (!one && blockIdx.x == 0) {
        const double sr = scalbn(1.0, er), sc = -scalbn(1.0, -eC);
        for (int e = threadIdx.x; e < 13 * 32; e += blockDim.x) {
            const int k = e / 32;
            const double2 v = (e & 31) <= Q ? tl_red[(size_t)j * 13 * 32 + e] : zero;
            red[(size_t)j * 13 * 32 + e] = coef(v, k < 10 ? 1.0 : (k == 10 ? sr : sc));
        }
    }
}

static bool fx_alloc(FactorSet& fs, int N, int nsteps, int batch) {
    const size_t S = fs.P + 1, ns = nsteps;
    bool ok = cudaMalloc(&fs.fx_sub, sizeof(FxSub) * N * ns) == cudaSuccess;
    ok &= cudaMalloc(&fs.fx_mx, swr_fx_bounds_bytes(N) * batch) == cudaSuccess;
    ok &= cudaMalloc(&fs.fx_rows, sizeof(int4) * ns * N * S * (4 * fs.L + 13)) == cudaSuccess;
    ok &= cudaMalloc(&fs.fx_red, sizeof(int4) * ns * N * 13 * 32) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        cudaFree(fs.fx_sub);
        cudaFree(fs.fx_mx);
        cudaFree(fs.fx_rows);
        cudaFree(fs.fx_red);
        fs.fx_sub = nullptr;
        fs.fx_mx = nullptr;
        fs.fx_rows = fs.fx_red = nullptr;
    }
    return ok;
}

size_t swr_fx_step_bytes(int N, int L, int P) {
    return sizeof(int4) * N * ((size_t)(P + 1) * (4 * L + 13) + 13 * 32) + sizeof(FxSub) * N;
}

int swr_fx_alloc_steps(FactorSet& fs, int N) {
    const size_t S = fs.P + 1;
    if (fs.nsteps < 2 || S >= kTlMaxSep) return -2;
    if (fs.fx_steps) return 0;
    if (!fs.tl_pcr && S > 32) {   // two-level data of one batch
        const size_t nb = fs.batch;
        bool ok = cudaMalloc(&fs.tl_pcr, sizeof(double2) * nb * N * 10 * S) == cudaSuccess;
        ok &= cudaMalloc(&fs.tl_aux, sizeof(double2) * nb * N * 3 * S) == cudaSuccess;
        ok &= cudaMalloc(&fs.tl_red, sizeof(double2) * nb * N * 13 * 32) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return -1;
        }
    }
    if (!fx_alloc(fs, N, fs.nsteps, fs.batch)) return -1;
    fs.fx_steps = true;
    return 0;
}

int swr_launch_fx_prepare(FactorSet& fs, int N, cudaStream_t s, int t0, int nb, double hist) {
    const int S = fs.P + 1, one = S <= 32;
    if (fs.nsteps > 1 ? !fs.fx_steps : (!one && (!fs.tl_ok || fs.tl_rs != 32))) return -2;
    if (!fs.fx_sub && !fx_alloc(fs, N, 1, 1)) return -1;
    const dim3 grid((S + 63) / 64, N, nb);
    if (cudaMemsetAsync(fs.fx_mx, 0, swr_fx_bounds_bytes(N) * nb, s) != cudaSuccess) return -1;
    const double2* fac = fs.fac + (size_t)t0 * fs.fstride;
    const double2* sep = fs.sep + (size_t)t0 * fs.sstride;
    const double2* pcr = fs.pcr + (size_t)t0 * fs.pstride;
    k_fx_bounds<<<grid, 64, 0, s>>>(fs.L, fs.P, fs.levels, one, fs.sub_P, fs.clen, fac, sep, pcr,
                                    fs.tl_pcr, fs.tl_aux, fs.tl_red, fs.fx_mx, fs.fstride,
                                    fs.sstride, fs.pstride);
    k_fx_convert<<<grid, 64, 0, s>>>(fs.L, fs.P, fs.levels, one, fs.sub_P, fs.clen, fac, sep, pcr,
                                     fs.tl_pcr, fs.tl_aux, fs.tl_red, fs.fx_mx,
                                     fs.fx_sub + (size_t)t0 * N,
                                     fs.fx_rows + (size_t)t0 * N * S * (4 * fs.L + 13),
                                     fs.fx_red + (size_t)t0 * N * 13 * 32, fs.fstride, fs.sstride,
                                     fs.pstride, hist);
    swr_count_launch(2);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// Scale of every system from its state after step 1 (u1, local node order at soff) and, for a
// driven march, its flux inputs, which are converted here: fin[q][side][t - 1] the term
// -l_t / (i kappa) of the end's row at the system's first scale.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_fx_start(const FxMarchArgs a, const double2* __restrict__ gin,
                                                  double2 inv_ik) {
    __shared__ unsigned long long mx, mf;
    __shared__ int ssc, sbad;
    const int q = blockIdx.x, j = a.sys[q].sub, n = a.sub_n[j];
    const MarchSys sy = a.sys[q];
    if (threadIdx.x == 0) mx = mf = 0;
    __syncthreads();
    unsigned long long m = 0, f = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double2 v = a.u1[a.soff[q] + i];
        m = max(m, (unsigned long long)__double_as_longlong(fabs(v.x)));
        m = max(m, (unsigned long long)__double_as_longlong(fabs(v.y)));
    }
    atomicMax(&mx, m);
    auto flux = [&](int side, int t) {   // t: 0-based step
        const int in = side ? sy.in_r : sy.in_l;
        if (in < 0 || !(a.sub_tc[j] & (1 << side))) return make_double2(0.0, 0.0);
        const double2 g = gin[(size_t)in + t];
        return cmul(make_double2(-g.x, -g.y), inv_ik);
    };
    if (a.fin && gin)
        for (int e = threadIdx.x; e < 2 * (sy.nt - 1); e += blockDim.x) {
            const double2 v = flux(e & 1, 1 + (e >> 1));
            f = max(f, (unsigned long long)__double_as_longlong(fabs(v.x)));
            f = max(f, (unsigned long long)__double_as_longlong(fabs(v.y)));
        }
    atomicMax(&mf, f);
    bool out = false;   // per-step factors: any step's out of range
    if (a.stream)
        for (int t = threadIdx.x; t < sy.nt; t += blockDim.x)
            out |= a.fsub[(size_t)(a.fstep0 + (a.frev ? -t : t)) * a.N + j].bad != 0;
    out = __syncthreads_or(out);
    if (threadIdx.x == 0) {
        double top = __longlong_as_double((long long)mx), tf = __longlong_as_double((long long)mf);
        int sc = 0, b = a.stream ? 0 : a.fsub[j].bad;
        b |= out;
        for (double v : {top, tf}) b |= !isfinite(v) || v > 1e250;
        if (top < 1e-280) top = 0.0;   // far tails of a packet: marched as zero
        if (tf < 1e-280) tf = 0.0;
        if (!b) {
            if (top > 0.0) sc = (a.fin ? 55 : 56) - ilogb(top);
            if (tf > 0.0) {   // a row takes flux terms up to 6 times the state limit
                const int s2 = 59 - ilogb(tf);
                sc = top > 0.0 ? min(sc, s2) : s2;
            }
        }
        a.scale[q] = ssc = sc;
        a.bad[q] = sbad = b;
    }
    __syncthreads();
    if (!a.fin || sbad || !gin) return;
    const double s1 = fx_pow2(ssc);
    FxC* fo = reinterpret_cast<FxC*>(a.fin) + (size_t)q * 2 * a.nt;
    for (int e = threadIdx.x; e < 2 * (sy.nt - 1); e += blockDim.x) {
        const int side = e & 1, t = 1 + (e >> 1);
        const double2 v = flux(side, t);
        fo[(size_t)side * a.nt + t] = FxC{__double2ll_rn(v.x * s1), __double2ll_rn(v.y * s1)};
    }
}

// ---------------------------------------------------------------------------
// The march: steps 2..nt of up to R right-hand sides of one subdomain per cluster of C CTAs
// (T threads per right-hand side and CTA; thread p = rank T + t owns separator p and chunk p).
// ONE: a system is one warp (C = 1, T = 32, at most 32 separators), PCR over its lanes.
// Otherwise the two-level separator solve of k_march_tl: each warp's super-separator row
// and its part of the next one go to every CTA of the cluster (A[q], B[q], double-buffered by
// step), and every warp solves the reduced system.  Within a CTA the warps of a system meet at
// a named barrier; across a cluster the rows are pushed with st.async onto an mbarrier per
// right-hand side and step parity, so that systems sharing CTAs never wait for one another (a
// cluster barrier per step with rows read back through distributed shared memory: 13.3 ms for
// the N = 16 build of the scaling workload).
// When a component passes the trigger the whole system is scaled down by 4: in the same step
// if it is one warp, one step later otherwise, the word travelling in a spare bit of A.  End
// traces (and through them the recorded states) carry the shift of their step.
// FLUX: flux inputs (a.fin).  HIST: S_0^2 ends.  STREAM: per-step factors.  FULL: the products of
// the low limbs too, everywhere (coarse grids and S_0^2 ends, see plan_create).
// Shared memory: a row of coefficients per chunk, once for all R (its odd length in 16-byte
// units keeps a warp's reads free of bank conflicts), the reduced system, A and B.
// ---------------------------------------------------------------------------
constexpr int kFxHist = 1;    // history sums are kept in units of 2^kFxHist
constexpr int kFxSlots = 34;   // A / B entries per right-hand side and parity

__device__ __forceinline__ unsigned fx_saddr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned fx_mapa(unsigned addr, int cta) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}
__device__ __forceinline__ void fx_push(unsigned addr, unsigned mbar, FxC x) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "l"(x.r), "l"(x.i), "r"(mbar) : "memory");
}
// wait for the phase of this parity; false after `polls` polls of up to a microsecond (a million:
// about a second; the caller flags a timeout)
__device__ __forceinline__ bool fx_wait(unsigned mbar, unsigned parity, int polls) {
    for (int k = 0; k < polls; ++k) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred q;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2, 1000;\n\t"
                     "selp.u32 %0, 1, 0, q;\n\t}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// S_0^2 history of one end, sum_{s<t} beta_{t-s} v_s, by one full warp in units of 2^kFxHist:
// lanes strided over s, a fixed butterfly (every lane gets the sum).  v_0, v_1 in registers, v_s
// at tr[s - 1] with its shift; the current shift is sh.
__device__ __forceinline__ FxC fx_history(const int2* __restrict__ beta, FxC v0, FxC v1,
                                          const FxC* tr, const int* tsh, int t, int sh, int lane) {
    fx_int hr = 0, hi = 0, mr = 0, mi = 0;
#pragma unroll 1
    for (int s = lane; s < t; s += 32) {
        const FxC x = s == 0 ? v0 : (s == 1 ? v1 : tr[s - 1]);
        const int k = sh - (s < 2 ? 0 : tsh[s - 1]);
        const fx_int half = ((fx_int)1 << k) >> 1;
        const FxS f = fx_split(FxC{(x.r + half) >> k, (x.i + half) >> k});
        const int2 b = beta[t - s];
        hr = fx_mw(f.rh, b.x, hr);
        hi = fx_mw(f.ih, b.x, hi);
        mr = fx_mw(f.rl, b.x, fx_mw(f.rh, b.y, mr));
        mi = fx_mw(f.il, b.x, fx_mw(f.ih, b.y, mi));
        mr += __mulhi(f.rl, b.y);
        mi += __mulhi(f.il, b.y);
        hr += mr >> 32;
        hi += mi >> 32;
        mr &= 0xffffffffLL;
        mi &= 0xffffffffLL;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        hr += __shfl_xor_sync(0xffffffffu, hr, off);
        hi += __shfl_xor_sync(0xffffffffu, hi, off);
        mr += __shfl_xor_sync(0xffffffffu, mr, off);
        mi += __shfl_xor_sync(0xffffffffu, mi, off);
    }
    // (H 2^64 + M 2^32) / 2^61 / 2^kFxHist.  sum |beta_s| < 72 for 2048 steps and |v| < 2^58, so
    // that a sum may reach 1.12 2^63; one that wraps is then below -2^60 or above 2^60, where the
    // march's range check of the history flags the system.  (H itself stays below 2^62.)
    constexpr int e = 29 + kFxHist;
    const fx_int half = (fx_int)1 << (e - 1);
    const FxC a = {(hr << (3 - kFxHist)) + ((mr + half) >> e), (hi << (3 - kFxHist)) + ((mi + half) >> e)};
    return a;
}

template <int L, bool ONE, bool FLUX, bool STREAM, bool HIST, bool FULL>
__global__ void __launch_bounds__(L == 16 ? 256 : (L == 4 && !STREAM ? 512 : 384), 1)
    k_march_fx(const FxMarchArgs a) {
    constexpr int ROW = 4 * L + 13;
    constexpr int KT = FLUX ? 24 : 25;   // the trigger is 2^(32 + KT)
    extern __shared__ int4 fsm[];
    const int T = ONE ? 32 : a.T, C = ONE ? 1 : a.C, R = a.R, P = a.P, S = P + 1;
    const int RD = ONE ? 0 : 13 * 32;
    const int BUF = ROW * T + RD;         // rows, then the reduced system [13][32]; STREAM: two
    const int4* srd = fsm + ROW * T;
    FxC* sA = reinterpret_cast<FxC*>(fsm + (STREAM ? 2 : 1) * BUF);  // [2][R][kFxSlots]
    FxC* sB = sA + (ONE ? 0 : 2 * R * kFxSlots);
    unsigned long long* mbar =
        reinterpret_cast<unsigned long long*>(sB + (ONE ? 0 : 2 * R * kFxSlots));   // [2][R]
    unsigned long long* full = mbar + 2 * R;   // STREAM: [2] a buffer's rows are there
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (!ONE && C > 1) ? (int)cl.block_rank() : 0;
    const int tid = threadIdx.x, lane = tid & 31;
    const int r = tid / T, t0 = tid - r * T;
    const int p = rank * T + t0;
    const int* grp = a.grp + (size_t)(ONE ? blockIdx.x : blockIdx.x / C) * R;
    int first = -1;
    for (int k = 0; k < R; ++k)
        if (grp[k] >= 0) first = grp[k];
    const int j = a.sys[first].sub;
    const int Pj = a.sub_P[j], Q = (Pj + 31) >> 5;
    FxSub f = a.fsub[(size_t)(STREAM ? a.fstep0 : 0) * (STREAM ? a.N : 0) + j];
    const int have = max(0, min(T, S - rank * T)) * ROW;
    // rows of the separators this CTA holds (one contiguous piece), zero beyond them.  STREAM:
    // step t's rows and reduced system go to buffer t & 1 by one bulk copy each
    auto fetch = [&](int t) {
        if (j == a.withhold) return;   // false but under the test hook
        const size_t st = a.fstep0 + (a.frev ? 1 - t : t - 1);
        const unsigned dst = fx_saddr(fsm + (t & 1) * BUF), mb = fx_saddr(full + (t & 1));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                     "r"(16u * (have + RD)) : "memory");
        if (have)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(dst), "l"(a.rows + ((st * a.N + j) * S + rank * T) * ROW),
                         "r"(16u * have), "r"(mb) : "memory");
        if (RD)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(dst + 16u * ROW * T), "l"(a.red + (st * a.N + j) * RD), "r"(16u * RD),
                         "r"(mb) : "memory");
    };
    if (STREAM) {
        for (int e = tid; e < 2 * BUF; e += blockDim.x) fsm[e] = make_int4(0, 0, 0, 0);
        if (tid < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fx_saddr(full + tid)) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    } else {
        const int4* src = a.rows + ((size_t)j * S + rank * T) * ROW;
        for (int e = tid; e < ROW * T; e += blockDim.x) fsm[e] = e < have ? src[e] : make_int4(0, 0, 0, 0);
        if (!ONE)
            for (int e = tid; e < RD; e += blockDim.x) fsm[ROW * T + e] = a.red[(size_t)j * RD + e];
    }
    if (!ONE) {
        for (int e = tid; e < 4 * R * kFxSlots; e += blockDim.x) sA[e] = fx_zero();
        if (C > 1 && tid < 2 * R) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fx_saddr(mbar + tid)) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    const int4* row = fsm + t0 * ROW;

    const int sidx = grp[r];
    const bool act = sidx >= 0 && !a.bad[max(sidx, 0)];     // uniform over the system
    const bool valid = act && p <= Pj;
    const MarchSys sy = a.sys[max(sidx, 0)];
    const int tcf = a.sub_tc[j];
    const int sp = valid ? a.sep_pos[j * S + p] : 0;
    const int nv = L - ((valid && p < Pj) ? a.clen[j * P + p] : 0);   // slots before the first node
    const int nvmax = L - (a.sub_n[j] - 1 - Pj) / Pj;                  // most of a chunk of j
    const int q = p >> 5;
    const int m = (32 * q < Pj) ? min(31, Pj - 1 - 32 * q) : 0;
    const bool member = !ONE && valid && lane >= 1 && lane <= m;
    const bool le = p == 0, re = p == Pj;
    // constants that round the shifts to nearest; ties (one in 2^k values) go up in odd steps
    // and down in even ones, so that they leave no mean behind
    int dd, ds2, one_s;   // one_s: 2^-s as a high limb
    fx_int half_2, half_z, half_d;
    auto scales = [&]() {
        dd = f.sd - f.s2;
        ds2 = f.s2 - f.s;
        half_2 = f.s2 ? (fx_int)1 << (f.s2 - 1) : 0;
        half_z = ds2 ? (fx_int)1 << (ds2 - 1) : 0;
        half_d = dd ? (fx_int)1 << (dd - 1) : 0;
        one_s = 1 << (29 - f.s);
    };
    scales();
    const int sc = act ? a.scale[sidx] : 0;
    FxC u[L], us = fx_zero(), usup = fx_zero();
    {
        const double2* u1 = a.u1 + (act ? a.soff[sidx] : 0);
        const double s1 = fx_pow2(sc);
        auto get = [&](int node) {
            const double2 v = u1[node];
            return FxC{__double2ll_rn(v.x * s1), __double2ll_rn(v.y * s1)};
        };
#pragma unroll
        for (int i = 0; i < L; ++i) u[i] = valid ? get(i < nv ? sp : sp + 1 + i - nv) : fx_zero();
        if (valid) us = get(sp);
        if (!ONE && act && lane <= Q) usup = get(a.sep_pos[j * S + (lane < Q ? 32 * lane : Pj)]);
    }
    const bool rec = !FLUX && valid && a.urec && (sy.flags & SYS_REC_U);
    const int Sj = Pj + 1;
    FxC* ru = reinterpret_cast<FxC*>(a.urec) + (rec ? sy.rec : 0) + p;   // chunk-slot order
    auto record = [&]() {
#pragma unroll
        for (int i = 0; i < L; ++i)
            __stcs(reinterpret_cast<int4*>(ru + i * Sj), *reinterpret_cast<int4*>(&u[i]));
        __stcs(reinterpret_cast<int4*>(ru + L * Sj), *reinterpret_cast<int4*>(&us));
        ru += (L + 1) * Sj;
    };
    if (rec) record();
    FxC* tr = nullptr;   // end trace of this thread's separator, its flux input, its shifts
    const FxC* fin = nullptr;
    int* tsh = nullptr;
    int sh = 0;
    if (valid && ((le && (tcf & 1)) || (re && (tcf & 2)))) {
        const size_t o = ((size_t)sidx * 2 + (le ? 0 : 1)) * a.nt;
        tr = reinterpret_cast<FxC*>(a.trace) + o;
        tsh = a.tshift + o;
        tsh[0] = 0;
        if (FLUX && (le ? sy.in_l : sy.in_r) >= 0 && a.driven)
            fin = reinterpret_cast<const FxC*>(a.fin) + o;
    }
    unsigned mu = 0, mv = 0;
    bool grown = false, late = false;
    int tlate = 0;   // STREAM: the step whose wait ran out
    const int nw = Pj / 32 + 1;            // warps of the system that hold separators
    // CTAs of the cluster that do (none to push to under the test hook)
    const int ncta = j == a.withhold ? 0 : Pj / T + 1;
    // bytes a step pushes to each of them: A[0..Q], and B of every warp whose lane 31 is not
    // the system's last separator
    const unsigned txb = 16u * (Q + 1 + nw - ((Pj & 31) == 31 ? 1 : 0));
    if (!ONE && C > 1) cl.sync(); else __syncthreads();
    // a warp without separators of its own takes no part (its system's barrier counts it)
    const int nsteps = (act && (C == 1 || q < nw)) ? sy.nt : 0;
    // S_0^2: the warps that hold an end form its history; v_0 = u_0 and v_1 = (u_1 + u_0) / 2
    const bool hist = HIST && act;
    FxC v0 = fx_zero(), v1 = fx_zero();
    if (hist && tr) {
        const double s1 = fx_pow2(sc);
        const double2 z = (sy.flags & SYS_ZERO_U0) ? make_double2(0.0, 0.0)
                                                   : a.u0[a.sub_goff[j] + (le ? 0 : a.sub_n[j] - 1)];
        if (fabs(z.x * s1) < 2.8e17 && fabs(z.y * s1) < 2.8e17) {   // 2^58
            v0 = FxC{__double2ll_rn(z.x * s1), __double2ll_rn(z.y * s1)};
            v1 = FxC{(us.r + v0.r) >> 1, (us.i + v0.i) >> 1};
        } else {
            mu = 0x80000000u;
        }
    }
    FxC fnext = (FLUX && fin && nsteps > 1) ? fin[1] : fx_zero();
    // STREAM (one right-hand side per CTA): a CTA whose warps all sit out fetches nothing
    if (STREAM && tid == 0 && nsteps > 1) fetch(2);
#pragma unroll 1
    for (int t = 2; t <= nsteps; ++t) {
        if (STREAM) {
            f = a.fsub[(size_t)(a.fstep0 + (a.frev ? 1 - t : t - 1)) * a.N + j];
            scales();
            row = fsm + (t & 1) * BUF + t0 * ROW;
            srd = fsm + (t & 1) * BUF + ROW * T;
            if (ONE) {
                __syncwarp();   // the other buffer has been read
                if (tid == 0 && t < nsteps) fetch(t + 1);
            }
            late = !fx_wait(fx_saddr(full + (t & 1)), ((t - 2) >> 1) & 1, a.polls);
            late = __any_sync(0xffffffffu, late);
            // a system of several warps in one CTA gives up together, at the step's barrier
            if (late && (ONE || C > 1 || T == 32)) {
                tlate = t;
                break;
            }
        }
        const int tie = (t & 1) - 1;
        const fx_int r2 = half_2 + (f.s2 ? tie : 0), rz = half_z + (ds2 ? tie : 0);
        const fx_int rd = half_d + (dd ? tie : 0);
        const int par = t & 1;
        if (!ONE && C > 1 && t0 == 0)   // arm this CTA's barrier of the step
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                             fx_saddr(mbar + par * R + r)), "r"(txb) : "memory");
        FxC hb = fx_zero();   // this end's history sum
        if (hist) {
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
                if (!(tcf & (1 << side)) || q != (side ? Pj >> 5 : 0)) continue;   // uniform per warp
                const int el = side ? Pj & 31 : 0;
                const size_t o = ((size_t)sidx * 2 + side) * a.nt;
                const FxC h = fx_history(a.beta, fx_from(v0, el), fx_from(v1, el),
                                         reinterpret_cast<const FxC*>(a.trace) + o, a.tshift + o, t,
                                         sh, lane);
                if (lane == el && (side ? re : le)) {
                    hb = h;
                    reinterpret_cast<FxC*>(a.htrace)[o + t - 1] = h;
                }
            }
        }
        // ---- forward: right-hand sides, elimination, left-end functional ------------------
        FxC uR = fx_down(us, 1);
        if (!ONE) {
            const FxC x = fx_from(usup, q + 1);
            if (lane == 31) uR = x;
        }
        FxC z[L], dot = fx_zero(), uf = u[0];
        FxAcc da = fx_acc();
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const FxC l = i ? u[i > 0 ? i - 1 : 0] : us, rr = i + 1 < L ? u[i + 1 < L ? i + 1 : 0] : uR;
            const FxC fi = {4 * u[i].r + (l.r + rr.r), 4 * u[i].i + (l.i + rr.i)};
            const FxS fs = fx_split(fi);
            FxAcc c = fx_acc();
            fx_mac_pow2(c, fs, one_s);
            if (i) fx_mul<FULL>(c, fx_split(z[i > 0 ? i - 1 : 0]), row[4 * (i > 0 ? i - 1 : 0) + 1]);
            z[i] = fx_res(c);
            fx_mul<FULL>(da, fs, row[4 * i + 2]);
            if (i & 1) {   // |f| < 2^61: at most four products between foldings
                dot = fx_add(dot, fx_res(da));
                da = fx_acc();
            }
        }
        if (nvmax > 0) {
            uf = fx_sel(nv == 1, u[1], uf);
            if (nvmax > 1) {   // short systems only
#pragma unroll
                for (int i = 2; i < L; ++i) uf = fx_sel(nv == i, u[i], uf);
            }
        }
        // ---- separator right-hand sides --------------------------------------------------
        FxC cr, d;   // cr: this chunk's part of its right separator's row
        {
            FxAcc c = fx_acc();
            fx_mul<FULL>(c, fx_split(z[L - 1]), row[4 * (L - 1) + 1]);
            cr = fx_add(fx_shr_c(u[L - 1], f.s2, r2), fx_shr_c(fx_res(c), ds2, rz));
            FxC fo = (le || re) ? FxC{2 * us.r, 2 * us.i} : FxC{4 * us.r, 4 * us.i};
            if (!re) fo = fx_add(fo, uf);
            if (FLUX && fin) {
                fo = fx_add(fo, fx_shr(fnext, sh));
                if (t < nsteps) fnext = fin[t];
            }
            d = fx_add(fx_shr_c(fo, f.s2, r2), dot);
            const FxC cl_ = fx_up(cr, 1);
            if (lane > 0 && !le) d = fx_add(d, cl_);
            if (hist) {
                const int kh = f.s2 - a.c2e - kFxHist;
                FxAcc h = fx_acc_shr(kh);
                fx_mac_full(h, fx_split(hb), a.c2);
                d = fx_add(d, fx_res_shr(h, kh, mv, 60));
                mv |= fx_range<28>(0u, d) >> 2;
                mv |= fx_range<28>(0u, hb) >> 2;
            }
            if (!valid) d = fx_zero();
        }
        const FxC drow = d;
        d = fx_shr_c(d, dd, rd);
        mv |= fx_range<28>(0u, d) >> 2;
        // ---- PCR over the lanes -----------------------------------------------------
#pragma unroll 1
        for (int k = 0; k < 5; ++k) {
            const int st = 1 << k;
            const FxS ds = fx_split(d);
            FxS dm, dp;
            dm.rh = __shfl_up_sync(0xffffffffu, ds.rh, st);
            dm.rl = __shfl_up_sync(0xffffffffu, ds.rl, st);
            dm.ih = __shfl_up_sync(0xffffffffu, ds.ih, st);
            dm.il = __shfl_up_sync(0xffffffffu, ds.il, st);
            dp.rh = __shfl_down_sync(0xffffffffu, ds.rh, st);
            dp.rl = __shfl_down_sync(0xffffffffu, ds.rl, st);
            dp.ih = __shfl_down_sync(0xffffffffu, ds.ih, st);
            dp.il = __shfl_down_sync(0xffffffffu, ds.il, st);
            FxAcc c = fx_acc();
            fx_mul<FULL>(c, dm, row[4 * L + 2 * k]);
            fx_mul<FULL>(c, dp, row[4 * L + 2 * k + 1]);
            d = fx_add(d, fx_res(c));
            mv |= fx_range<28>(0u, d) >> 2;   // to the bit of fx_range<26>
        }
        FxC v;
        {
            FxAcc c = fx_acc_shr(f.kv);
            fx_mac_full(c, fx_split(d), row[4 * L + 10]);
            v = fx_res_shr(c, f.kv, mv);
        }
        FxC vR;
        bool down = false;   // scale the system down at the end of this step
        if (ONE) {
            mv = fx_range<26>(mv, v);
            vR = fx_down(v, 1);
        } else {
            // ---- reduced system: A[q] = row of super-separator q as far as warp q knows it,
            // B[q + 1] = this warp's part of the next row ------------------------------------
            if (member) mv = fx_range<26>(mv, v);
            const FxC yf = fx_from(v, 1), yl = fx_from(v, m);
            {
                const bool own_last = re && lane != 0;   // row Pj within this warp
                const int qi = own_last ? Q : (lane == 31 ? q + 1 : q);
                const bool up = lane == 0 && !re;        // couples to the first of its own chunk
                FxC y = up ? yf : yl;
                if (m == 0 || (lane == 0 && re)) y = fx_zero();
                FxAcc c = fx_acc_shr(f.kc);
                fx_mul<FULL>(c, fx_split(y), srd[(up ? 12 : 11) * 32 + (qi & 31)]);
                const FxC mine = (lane == 31 && !own_last) ? cr : drow;
                FxC x = fx_add(fx_shr(mine, f.sr - f.s2), fx_res_shr(c, f.kc, mv, 60));
                const bool isA = lane == 0 || own_last, isB = lane == 31 && !own_last;
                if (isB && p >= Pj) x = fx_zero();
                if (isA || isB) mv |= fx_range<28>(0u, x) >> 2;
                if (lane == 0 && grown) x.r ^= (fx_int)1 << 62;   // the state has passed the trigger
                if ((isA && valid) || (isB && q < nw)) {
                    FxC* dst = (isA ? sA : sB) + (par * R + r) * kFxSlots + qi;
                    if (C == 1) {
                        *dst = x;
                    } else {
                        const unsigned da_ = fx_saddr(dst), mb = fx_saddr(mbar + par * R + r);
                        for (int cta = 0; cta < ncta; ++cta) fx_push(fx_mapa(da_, cta), fx_mapa(mb, cta), x);
                    }
                }
            }
            if (C > 1) {
                late = !fx_wait(fx_saddr(mbar + par * R + r), ((t - 2) >> 1) & 1, a.polls);
                if (__any_sync(0xffffffffu, late)) {   // give up; a last bounded wait for rows in flight
                    late = true;
                    fx_wait(fx_saddr(mbar + par * R + r), ((t - 2) >> 1) & 1, a.polls);
                    break;
                }
            } else if (STREAM && T > 32) {
                // with the warps' late flags: one that left its loop alone would leave the others
                // at this barrier without a limit (the rows it worked on are not there, so what
                // it put into A and B is never used)
                int any;
                asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\t"
                             "barrier.cta.red.or.pred q, %1, %2, q;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                             : "=r"(any) : "r"(r + 1), "r"(T), "r"((int)late) : "memory");
                if (any) {
                    late = true;
                    tlate = t;
                    break;
                }
            } else if (T > 32) {
                asm volatile("bar.sync %0, %1;" ::"r"(r + 1), "r"(T) : "memory");
            } else {
                __syncwarp();
            }
            // every warp has pushed this step's rows, so it has read the last step's buffer
            if (STREAM && tid == 0 && t < nsteps) fetch(t + 1);
            FxC x = fx_zero();
            if (lane <= Q) {
                x = sA[(par * R + r) * kFxSlots + lane];
                down = ((x.r >> 62) ^ (x.r >> 63)) & 1;
                x.r = (fx_int)((unsigned long long)x.r << 2) >> 2;
                if (lane > 0 && (lane < Q || (Pj & 31) == 0))
                    x = fx_add(x, sB[(par * R + r) * kFxSlots + lane]);
            }
            down = __any_sync(0xffffffffu, down);
#pragma unroll 1
            for (int k = 0; (1 << k) <= Q; ++k) {   // no coupling beyond: uniform over the system
                const int st = 1 << k;
                const FxC xm = fx_up(x, st), xp = fx_down(x, st);
                FxAcc c = fx_acc();
                mv |= fx_range<28>(0u, x) >> 2;
                fx_mul<FULL>(c, fx_split(xm), srd[(2 * k) * 32 + lane]);
                fx_mul<FULL>(c, fx_split(xp), srd[(2 * k + 1) * 32 + lane]);
                x = fx_add(x, fx_res(c));
            }
            mv |= fx_range<28>(0u, x) >> 2;
            {
                FxAcc c = fx_acc_shr(f.kr);
                fx_mac_full(c, fx_split(x), srd[10 * 32 + lane]);
                x = fx_res_shr(c, f.kr, mv);
            }
            if (lane > Q) x = fx_zero();
            mv = fx_range<26>(mv, x);
            usup = fx_twice_less(x, usup);
            const FxC xq = fx_from(x, q), xn = fx_from(x, q + 1), xQ = fx_from(x, Q);
            FxAcc c = fx_acc();
            fx_mac_full(c, fx_split(xq), row[4 * L + 11]);
            fx_mac_full(c, fx_split(xn), row[4 * L + 12]);
            v = member ? fx_add(v, fx_res(c)) : (re ? xQ : xq);
            if (!valid) v = fx_zero();
            vR = fx_down(v, 1);
            if (lane == 31) vR = xn;
        }
        // ---- backward: chunk values, Crank-Nicolson update --------------------------------
        unsigned ms = 0;
        {
            const FxS vl = fx_split(v);
            FxS xs = fx_split(vR);
#pragma unroll
            for (int i = L - 1; i >= 0; --i) {
                FxAcc c = fx_acc();
                fx_mul<FULL>(c, fx_split(z[i]), row[4 * i]);
                fx_mul<FULL>(c, vl, row[4 * i + 3]);
                fx_mul<FULL>(c, xs, row[4 * i + 1]);
                const FxC x = fx_res(c);
                xs = fx_split(x);
                u[i] = fx_twice_less(x, u[i]);
                ms = fx_range<KT>(ms, u[i]);
            }
        }
        us = fx_twice_less(v, us);
        ms = fx_range<KT>(ms, us);
        if (tr) {
            tr[t - 1] = v;
            tsh[t - 1] = sh;
        }
        if (hist) __syncwarp();   // the next step's history reads them
        if (rec) record();
        const bool pass = __any_sync(0xffffffffu, ms >> (KT + 1));   // beyond the trigger
        if (pass) {
#pragma unroll
            for (int i = 0; i < L; ++i) mu = fx_range<26>(mu, u[i]);
            mu = fx_range<26>(mu, us);
        }
        if (ONE)
            down = pass;
        else
            grown = pass && !down;   // the next step's word; not of a state that is scaled down now
        if (down) {
#pragma unroll
            for (int i = 0; i < L; ++i) u[i] = fx_shr_c(u[i], 2, 2);
            us = fx_shr_c(us, 2, 2);
            usup = fx_shr_c(usup, 2, 2);
            sh += 2;
            if (sh > 900) mu = 0x80000000u;
        }
    }
    if (valid && ((mu >> 27) || (mv >> 27) || late)) a.bad[sidx] = 1;
    if (late) atomicOr(a.status, ST_TIMEOUT);
    if (STREAM && tlate && tid == 0) {   // copies in flight, once more within the limit
        fx_wait(fx_saddr(full + (tlate & 1)), ((tlate - 2) >> 1) & 1, a.polls);
        if (ONE && tlate < nsteps)
            fx_wait(fx_saddr(full + ((tlate + 1) & 1)), ((tlate - 1) >> 1) & 1, a.polls);
    }
    if (valid && (sy.flags & (SYS_REC_LAST | SYS_WRITE_UT))) {
        const double s1 = fx_pow2(sh - sc);
        double2* last = (sy.flags & SYS_REC_LAST) && a.urec ? a.urec + sy.rec : nullptr;
        double2* uT = (sy.flags & SYS_WRITE_UT) && a.uT ? a.uT + a.sub_goff[j] : nullptr;
        auto put = [&](int node, FxC x, bool mine) {
            const double2 o = make_double2((double)x.r * s1, (double)x.i * s1);
            if (last) last[node] = o;
            if (uT && mine) uT[node] = o;
        };
#pragma unroll
        for (int i = 0; i < L; ++i)
            if (i >= nv) put(sp + 1 + i - nv, u[i], true);
        put(sp, us, sp > 0 || !(tcf & 1));   // an interface node belongs to the left subdomain
    }
    // keep this CTA's shared memory alive until every CTA of the cluster is done
    if (!ONE && C > 1) cl.sync();
}

// Fluxes of steps 2..nt from the integer end traces (and the traces themselves for SYS_TRACE);
// one CTA per system.  A trace keeps its absolute error, a few units, however small it is: an
// impulse march with a trace that never reaches 2^40 units (2^-16 of the state), and any other
// march with no trace (nor flux input) that does, are flagged for FP64 instead.
__global__ void __launch_bounds__(128) k_fx_flux(const FxMarchArgs a, double2 two_sigma,
                                                 const double2* __restrict__ gin,
                                                 double2* __restrict__ gout,
                                                 double2* __restrict__ vtrace) {
    const int q = blockIdx.x, ntmax = a.nt;
    const MarchSys sy = a.sys[q];
    const int tcf = a.sub_tc[sy.sub];
    if (a.bad[q]) return;
    const FxC* tr = reinterpret_cast<const FxC*>(a.trace) + (size_t)q * 2 * ntmax;
    const bool imp = sy.flags & (SYS_IMP_L | SYS_IMP_R);
    if (sy.nt > 1 && a.scale[q] != 0) {
        unsigned ml = 0, mr = 0;
        for (int t = 1 + threadIdx.x; t < sy.nt; t += blockDim.x) {
            if (tcf & 1) ml = fx_mag(ml, tr[t]);
            if (tcf & 2) mr = fx_mag(mr, tr[ntmax + t]);
            if (a.driven) {   // the flux update's own input
                const double big = scalbn(1.0, 40 - a.scale[q]);
                for (int in : {sy.in_l, sy.in_r})
                    if (in >= 0 && fmax(fabs(gin[(size_t)in + t].x), fabs(gin[(size_t)in + t].y)) >= big)
                        ml |= 256u;
            }
        }
        const bool bl = __syncthreads_or(ml >= 256u), br = __syncthreads_or(mr >= 256u);
        const bool hl = tcf & 1, hr = tcf & 2;
        if (imp ? (hl && !bl) || (hr && !br) : !bl && !br) {
            if (threadIdx.x == 0) a.bad[q] = 1;
            return;
        }
    }
    const double s0 = fx_pow2(-a.scale[q]);
    for (int e = threadIdx.x; e < 2 * (sy.nt - 1); e += blockDim.x) {
        const int side = e & 1, t = 1 + (e >> 1);
        const size_t o = (size_t)side * ntmax + t;
        if (!(tcf & (1 << side))) continue;
        const double s1 = s0 * fx_pow2(a.tshift[(size_t)q * 2 * ntmax + o]);
        const double2 v = make_double2((double)tr[o].r * s1, (double)tr[o].i * s1);
        const int out = side ? sy.out_b : sy.out_a, in = side ? sy.in_r : sy.in_l;
        if (out >= 0 && gout) {
            const double2 g = (in >= 0 && gin) ? gin[(size_t)in + t] : make_double2(0.0, 0.0);
            double2 o2 = csub(cmul(two_sigma, v), g);
            if (a.beta) {
                const FxC h = reinterpret_cast<const FxC*>(a.htrace)[(size_t)q * 2 * ntmax + o];
                const double s2 = s1 * (double)(1 << kFxHist);
                o2 = cfma(a.two_c2, make_double2((double)h.r * s2, (double)h.i * s2), o2);
            }
            gout[(size_t)out + t] = o2;
        }
        if ((sy.flags & SYS_TRACE) && vtrace) vtrace[(size_t)q * 2 * ntmax + o] = v;
    }
}

// ---------------------------------------------------------------------------
// Launch shape: chunk length, CTAs per subdomain and threads per right-hand side.
// ---------------------------------------------------------------------------
static int fx_smem_bytes(int L, int T, int R, bool one, bool stream) {
    int b = 16 * ((4 * L + 13) * T + (one ? 0 : 13 * 32)) * (stream ? 2 : 1) + 16 * R + 16;
    if (!one) b += 16 * 4 * R * kFxSlots;
    return b;
}

// (threads: what the registers of an instantiation allow; shared memory: 220 KB)
bool swr_fx_fits(int L, int T, int R, bool one, bool stream) {
    const int tmax = L == 16 ? 256 : (L == 4 && !stream ? 512 : 384);
    return R * T <= tmax && fx_smem_bytes(L, T, R, one, stream) <= 220 * 1024;
}

bool swr_fx_shape(int nmax, int ngroups, int R, int forceL, int nsm, FxShape* out, bool stream) {
    const int Ls[4] = {16, 12, 8, 4};
    double best = -1.0;
    for (int L : Ls) {
        if ((forceL && L != forceL) || (stream && L > 8)) continue;
        const int S = (nmax - 1 + L) / (L + 1) + 1;   // separators
        if (S >= kTlMaxSep) continue;
        for (int C = 1; C <= 16; ++C) {
            const bool one = S <= 32;
            const int T = ((S + C - 1) / C + 31) / 32 * 32;
            if ((one && C > 1) || !swr_fx_fits(L, T, R, one, stream) || (C > 1 && (C - 1) * T >= S)) continue;
            const int smem = fx_smem_bytes(L, T, R, one, stream);
            // cycles a warp's step costs its SM sub-partition, and its own length (measured: 5000
            // and 9700 for a one-warp system with L = 12; 9800 for L = 4 over a cluster)
            const double iss = 320.0 * L + (one ? 1200.0 : 2600.0);
            const double lat = 620.0 * L + (one ? 2300.0 : 5800.0) + (C > 1 ? 1500.0 : 0.0);
            const int regs = L == 16 ? 256 : (L == 4 && !stream ? 128 : 168);
            const int res = std::max(1, std::min(227 * 1024 / (smem + 1024), 65536 / (R * T * regs)));
            const double all = (double)ngroups * C;
            const double waves = std::ceil(all / ((double)nsm * res));
            const double ctas = std::min((double)res, std::ceil(all / nsm));
            const double warps = ctas * R * (T / 32) / 4.0;   // per SM sub-partition
            double step = waves * std::max(lat, std::max(warps, 1.0) * iss);
            // four-node chunks only where they are clearly faster: the factors of more separators
            // carry more rounding error, the same here and in FP64 (the build's columns of 20 drawn
            // problems of 5000 to 85000 nodes against extended precision: larger than with eight
            // nodes in 17, by 9 % in the mean; d and R g alike).  On 15 problems the factor chose
            // eight nodes twice where four were faster (14019 nodes in 28 subdomains, 150 steps: 1.29
            // against 1.09 ms a build; 76618 in 138: 1.32, 1.26).
            if (L == 4 && !stream) step *= 1.25;
            if (best < 0.0 || step < best) {
                best = step;
                *out = FxShape{L, C, T};
            }
        }
    }
    return best >= 0.0;
}

template <int L, bool ONE, bool FLUX, bool STREAM, bool HIST, bool FULL>
static int launch_fx_t(const FxMarchArgs& a, int ngroups, cudaStream_t s) {
    const int smem = fx_smem_bytes(L, a.T, a.R, ONE, STREAM);
    auto kern = k_march_fx<L, ONE, FLUX, STREAM, HIST, FULL>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return -1;
    // several CTAs share an SM: all of its shared memory
    if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return -1;
    if (a.C > 8 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return -1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ngroups * a.C);
    cfg.blockDim = dim3(a.T * a.R);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    swr_count_launch(1);
    return cudaLaunchKernelEx(&cfg, kern, a) == cudaSuccess ? 0 : -1;
}

template <int L, bool FLUX, bool STREAM, bool HIST>
static int launch_fx_f(const FxMarchArgs& a, bool one, bool full, int ngroups, cudaStream_t s) {
    if (full) return one ? launch_fx_t<L, true, FLUX, STREAM, HIST, true>(a, ngroups, s)
                         : launch_fx_t<L, false, FLUX, STREAM, HIST, true>(a, ngroups, s);
    if constexpr (HIST) return -2;
    else return one ? launch_fx_t<L, true, FLUX, STREAM, HIST, false>(a, ngroups, s)
                    : launch_fx_t<L, false, FLUX, STREAM, HIST, false>(a, ngroups, s);
}

template <int L>
static int launch_fx_l(const FxMarchArgs& a, bool one, int ngroups, cudaStream_t s) {
    const bool full = a.full;
    if constexpr (L <= 8) {   // per-step factors: latency bound, short chunks
        if (a.stream) return launch_fx_f<L, true, true, false>(a, one, full, ngroups, s);
    }
    if (a.stream) return -2;
    if (a.beta)   // S_0^2 ends: instantiations of their own, so that Robin ones keep their registers
        return a.fin ? launch_fx_f<L, true, false, true>(a, one, true, ngroups, s)
                     : launch_fx_f<L, false, false, true>(a, one, true, ngroups, s);
    return a.fin ? launch_fx_f<L, true, false, false>(a, one, full, ngroups, s)
                 : launch_fx_f<L, false, false, false>(a, one, full, ngroups, s);
}

int swr_launch_fx_start(const FactorSet& fs, FxMarchArgs a, int nsys, const double2* gin,
                        double2 inv_ik, cudaStream_t s) {
    a.fsub = fs.fx_sub;
    a.stream = fs.nsteps > 1;
    k_fx_start<<<nsys, 256, 0, s>>>(a, gin, inv_ik);
    swr_count_launch(1);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Test hook of the waits (swr_test_wait_hook): taken by the launches enqueued after it.
static std::atomic<long long> g_fx_polls{1000000};
static std::atomic<int> g_fx_withhold{-1};
void swr_fx_set_wait_hook(long long polls, int withhold) {
    g_fx_polls = polls > 0 ? std::min(polls, 1000000LL) : 1000000LL;
    g_fx_withhold = withhold;
}

int swr_launch_march_fx(const FactorSet& fs, FxMarchArgs a, int ngroups, cudaStream_t s) {
    a.polls = (int)g_fx_polls;
    a.withhold = g_fx_withhold;
    a.P = fs.P;
    a.sub_P = fs.sub_P;
    a.sep_pos = fs.sep_pos;
    a.clen = fs.clen;
    a.fsub = fs.fx_sub;
    a.rows = fs.fx_rows;
    a.red = fs.fx_red;
    a.stream = fs.nsteps > 1;
    if (a.stream && (a.R != 1 || !a.fin)) return -2;
    const bool one = fs.P + 1 <= 32;
    if (one && (a.C != 1 || a.T != 32)) return -2;
    switch (fs.L) {
        case 4: return launch_fx_l<4>(a, one, ngroups, s);
        case 8: return launch_fx_l<8>(a, one, ngroups, s);
        case 12: return launch_fx_l<12>(a, one, ngroups, s);
        case 16: return launch_fx_l<16>(a, one, ngroups, s);
        default: return -2;
    }
}

int swr_launch_fx_flux(const FxMarchArgs& a, int nsys, double2 two_sigma, const double2* gin,
                       double2* gout, double2* vtrace, cudaStream_t s) {
    k_fx_flux<<<nsys, 128, 0, s>>>(a, two_sigma, gin, gout, vtrace);
    swr_count_launch(1);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// u(T) by superposition of the recorded states (see k_superpose in swr_krylov.cu), for plans
// whose build marches ran here: one thread per recorded entry (chunk-slot order), the states
// read as integers and the fluxes of a side, times the scaling-down of the state each meets,
// held as limbs scaled by their largest component, |g| < 2^eg, C = g 2^(cb - eg).  With
// |X| <= 2^58 and cb = 56 (less for
// nt > 512) the high sums stay below 2^62 over all steps; the middle sums are folded into
// them every four steps.  A side marched in FP64 (flagged) is read as doubles in node order.
//
// Bound by memory: 0.80 ms for 3.2 GB of states (200001 nodes, 500 steps, 500 subdomains), with
// eight states of a thread in flight (each used as it arrives: 1.2 ms).  The FP64 form, its pipe
// at 97 %, takes 1.5 ms.
// ---------------------------------------------------------------------------
constexpr int kSupTile = 128;

template <bool FULL>
__device__ __forceinline__ double2 superpose_side_fx(const FxC* __restrict__ col, size_t stride,
                                                     bool in, const double2* __restrict__ gs,
                                                     int nt, int sc, const int* __restrict__ sh, int4* tile,
                                                     unsigned long long* mx) {
    unsigned long long m = 0;
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
        const double up = fx_pow2(sh[nt - 1 - t]);
        m = max(m, (unsigned long long)__double_as_longlong(fabs(gs[t].x * up)));
        m = max(m, (unsigned long long)__double_as_longlong(fabs(gs[t].y * up)));
    }
    __syncthreads();
    if (threadIdx.x == 0) *mx = 0;
    __syncthreads();
    atomicMax(mx, m);
    __syncthreads();
    const double top = __longlong_as_double((long long)*mx);
    if (!(top > 0.0)) return make_double2(top, top);   // no flux (or NaN, which reaches u(T))
    if (!isfinite(top)) return make_double2(top, top);
    const int eg = ilogb(top) + 1;
    int lg = 9;
    while ((1 << lg) < nt) ++lg;
    const int cb = 56 - (lg - 9);
    fx_int hr = 0, hi = 0, mr = 0, mi = 0;
    for (int k0 = 0; k0 < nt; k0 += kSupTile) {
        const int kc = min(kSupTile, nt - k0);
        __syncthreads();
        for (int q = threadIdx.x; q < kSupTile; q += blockDim.x) {
            int4 c = make_int4(0, 0, 0, 0);
            if (q < kc) {   // Phi(k) multiplies the flux of step nt - k + 1
                const double2 g = gs[nt - 1 - (k0 + q)];
                // |g| 2^-eg < 1; fx_coef scales by 2^61
                const int e = cb - 61 - eg + sh[k0 + q];
                c = fx_coef(scalbn(g.x, e), scalbn(g.y, e));
            }
            tile[q] = c;
        }
        __syncthreads();
        if (!in) continue;
        const int4* pc = reinterpret_cast<const int4*>(col + (size_t)k0 * stride);
        // eight states in flight per thread (loaded before any is used), folded every four
        for (int q = 0; q < kc; q += 8) {
            int4 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[e] = __ldcs(pc + (size_t)min(q + e, kc - 1) * stride);   // past the end: times zero
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                FxAcc c = {hr, mr, hi, mi};
#pragma unroll
                for (int e = h; e < h + 4; ++e) {
                    FxC x;
                    x.r = (fx_int)(((unsigned long long)(unsigned)v[e].y << 32) | (unsigned)v[e].x);
                    x.i = (fx_int)(((unsigned long long)(unsigned)v[e].w << 32) | (unsigned)v[e].z);
                    fx_mul<FULL>(c, fx_split(x), tile[q + e]);
                }
                hr = c.hr + (c.mr >> 32);
                hi = c.hi + (c.mi >> 32);
                mr = c.mr & 0xffffffffLL;
                mi = c.mi & 0xffffffffLL;
            }
        }
    }
    // X C = H 2^64 + M 2^32, of scale 2^(sc + cb - eg)
    const int e = sc + cb - eg;
    return make_double2(scalbn((double)hr, 64 - e) + scalbn((double)mr, 32 - e),
                        scalbn((double)hi, 64 - e) + scalbn((double)mi, 32 - e));
}

__device__ __forceinline__ double2 superpose_side_f64(const double2* __restrict__ col, size_t n,
                                                      bool in, const double2* __restrict__ gs,
                                                      int nt) {
    double2 acc = make_double2(0.0, 0.0);
    if (in)
        for (int k = 0; k < nt; ++k) acc = cfma(__ldcs(col + (size_t)k * n), gs[nt - 1 - k], acc);
    return acc;
}

template <bool FULL>
__global__ void __launch_bounds__(256) k_superpose_fx(
    int L, int P, const double2* __restrict__ urec, const long long* __restrict__ rec_base,
    const MarchSys* __restrict__ sys, const int3* __restrict__ subsys,
    const int* __restrict__ sub_n, const int* __restrict__ sub_goff,
    const int* __restrict__ sub_tc, const int* __restrict__ sub_P, const int* __restrict__ sep_pos,
    const unsigned char* __restrict__ clen, const int* __restrict__ scale,
    const int* __restrict__ shift, int ntmax, const int* __restrict__ bad, const double2* __restrict__ g, double2* __restrict__ uT) {
    __shared__ int4 tile[kSupTile];
    __shared__ unsigned long long mx;
    const int j = blockIdx.y, Sj = sub_P[j] + 1, n = sub_n[j];
    const int rs = (L + 1) * Sj, e = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x * blockDim.x >= rs) return;
    const int i = e / Sj, p = e - i * Sj;
    bool in = e < rs;
    int node = 0;
    if (in) {
        const int sp = sep_pos[j * (P + 1) + p];
        if (i == L) {
            node = sp;
        } else {
            const int nv = p < Sj - 1 ? L - clen[j * P + p] : L;   // slots before the first node
            in = i >= nv;
            node = sp + 1 + i - nv;
        }
    }
    const MarchSys sy = sys[j];
    const int nt = sy.nt;
    const double2* base = urec + rec_base[j];
    const int3 q = subsys[j];   // systems of the zero-flux march and the two impulses
    double2 u = in ? base[(size_t)2 * nt * rs + node] : make_double2(0.0, 0.0);
    for (int side = 0; side < 2; ++side) {
        const int s = side ? q.z : q.y, gi = side ? sy.in_r : sy.in_l;
        if (s < 0 || gi < 0) continue;
        const double2* col = base + (size_t)side * nt * rs;
        u = cadd(u, bad[s] ? superpose_side_f64(col + node, n, in, g + gi, nt)
                           : superpose_side_fx<FULL>(reinterpret_cast<const FxC*>(col) + e, rs, in, g + gi,
                                               nt, scale[s],
                                               shift + ((size_t)s * 2 + side) * ntmax, tile, &mx));
    }
    // the interface node belongs to the left subdomain
    if (in && !(node == 0 && (sub_tc[j] & 1))) uT[sub_goff[j] + node] = u;
}

int swr_launch_superpose_fx(const FactorSet& fs, const double2* urec, const long long* rec_base,
                            const MarchSys* sys, const int3* subsys, int N, const int* sub_n,
                            const int* sub_goff, const int* sub_tc, const int* scale,
                            const int* shift, int ntmax, const int* bad, const double2* g,
                            double2* uT, int full, cudaStream_t s) {
    dim3 grid(((fs.L + 1) * (fs.P + 1) + 255) / 256, N);
    const auto kern = full ? k_superpose_fx<true> : k_superpose_fx<false>;
    kern<<<grid, 256, 0, s>>>(fs.L, fs.P, urec, rec_base, sys, subsys, sub_n, sub_goff,
                                        sub_tc, fs.sub_P, fs.sep_pos, fs.clen, scale, shift, ntmax,
                                        bad, g, uT);
    swr_count_launch(1);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
