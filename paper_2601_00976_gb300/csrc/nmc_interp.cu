// opacity_interp: tetralinear interpolation of the EmAb / Iso log tables at
// arbitrary points (Sec. 2.3, tetralinear interpolation of chi_EmAb and the
// isoenergetic kernels).  One thread per point: uniform axes in
// (log10 rho, log10 T, Ye) give the cell directly, the energy axis (the node
// energies of the grid) is searched by bisection in log E; the 16 corner ln
// values are interpolated and exponentiated.  Two forms:
//  - fixed point (opacity_interp_fixed_kernel), for tables that fit Q53: the logarithms, the fifteen
//    linear interpolations and the exponential in 64-bit integers (nmc_fixed.cuh), two FP64
//    instructions per point (the Ye coordinate) instead of ~215.  Accuracy no worse: coordinates to
//    2^-52 of an octave, the interpolant to 2^-51 absolute, where FP64 rounds ln chi ~ -20 by
//    2^-49; against quad precision its error is 4-6 times smaller (5e-16 against 2.8e-15, 2-norm).
//    The sixteen corners come as four 32-byte cells (one L2 sector each).  4.0 M points: 1.37 ms in
//    FP64 (the FP64 pipe busy throughout), 0.166 ms in fixed point (24 G points/s).
//  - FP64 (opacity_interp_kernel), for any other table (an ln value of -infinity, say).
//
// opacity_interp_mixed: the same interpolation in FP32 on FP32 copies of the
// ln tables: FP32 logarithms, cell search and weights, the ln value as the
// first corner plus weighted differences (the corners are ~ -20, whose FP32
// sum would round ln chi by ~2e-6 in steps), and an FP32 exp; inputs and
// outputs stay FP64.  The energy axis is searched in a shared-memory copy of
// ln eps.  The table copy is regrouped per (T, rho, E) cell, eight corners to a
// 32-byte sector, so a point's 16 corner values come from two L2 sectors (from
// four with (rho, E) cells, which left the kernel at the L2's rate: 8.6 TB/s of
// sectors for 2.1 TB/s of points), and two points a thread are in flight.
// 8.4 M points: 0.168 ms before these and the integer conversions, 0.121 ms now
// (2.8 TB/s of points, 41% of the copy rate).  A context too short of memory for
// the cells reads the 16 values from the FP32 tables themselves: the same bits,
// 0.29 ms.
#include <cuda_runtime.h>
#include <math.h>

#include <cmath>
#include <string>
#include <vector>

#include "nmc_internal.h"
#include "nmc_eos.cuh"

namespace nmc {

namespace {

__device__ __forceinline__ void cell(double v, const Axis& ax, int* i, double* t) {
    double x = (v - ax.lo) * ax.inv_d;
    if (!(x >= 0.0)) x = 0.0;
    if (x > ax.n - 1) x = ax.n - 1;
    int c = (int)floor(x);
    if (c > ax.n - 2) c = ax.n - 2;
    *i = c;
    *t = x - c;
}

__global__ void opacity_interp_kernel(const DevGrid g, const DevTables tb, int which, int species,
                                      long long p, const double* __restrict__ rho,
                                      const double* __restrict__ T, const double* __restrict__ Ye,
                                      const double* __restrict__ E, double* __restrict__ out) {
    const double* tab = which == 0 ? tb.emab : tb.iso;
    const int NE = g.ne;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < p; i += (long long)gridDim.x * blockDim.x) {
        int ir, it, iy;
        double tr, tt, ty;
        cell(log10(rho[i]), tb.rho, &ir, &tr);
        cell(log10(T[i]), tb.t, &it, &tt);
        cell(Ye[i], tb.ye, &iy, &ty);
        // energy: ln E clamped to [ln eps_0, ln eps_{ne-1}], bisection for the cell
        double le = log(E[i]);
        if (!(le >= g.lneps[0])) le = g.lneps[0];
        if (le > g.lneps[NE - 1]) le = g.lneps[NE - 1];
        int lo = 0, hi = NE - 1;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (g.lneps[mid] <= le) lo = mid; else hi = mid;
        }
        const double te = (le - g.lneps[lo]) / (g.lneps[lo + 1] - g.lneps[lo]);
        const long long base = ((((long long)species * tb.ye.n + iy) * tb.t.n + it) * tb.rho.n + ir) * NE + lo;
        const long long dR = NE, dT = (long long)tb.rho.n * NE, dY = (long long)tb.t.n * tb.rho.n * NE;
        if (!NMC_IN_BOUNDS(g.dbg, base, tb.n_op, kDbgEmabIso) ||
            !NMC_IN_BOUNDS(g.dbg, base + dR + dT + dY + 1, tb.n_op, kDbgEmabIso))
            continue;
        double v = 0.0;
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) {
            const int ca = c8 & 1, cb = (c8 >> 1) & 1, cc = c8 >> 2;
            const double w = (ca ? tr : 1.0 - tr) * (cb ? tt : 1.0 - tt) * (cc ? ty : 1.0 - ty);
            const long long o = base + ca * dR + cb * dT + cc * dY;
            v += w * ((1.0 - te) * tab[o] + te * tab[o + 1]);
        }
        out[i] = exp(v);
    }
}

// Energy search of both forms.  A bisection is five or six dependent shared-memory loads; instead the
// logarithm's position on [lo, hi] picks one of kBuckets entries that hold the cell one bucket below
// (never above the right cell), and a short scan ends at the last cell whose lower node is <= le.
constexpr int kBuckets = 256;   // the kernels' block size

template <typename V>
__device__ __forceinline__ int cell_by_bisection(const V* node, int ne, V le) {
    int lo = 0, hi = ne - 1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (node[mid] <= le) lo = mid; else hi = mid;
    }
    return lo;
}

template <typename V>
__device__ __forceinline__ int cell_from(const V* node, int ne, V le, int lo) {
    while (lo < ne - 2 && node[lo + 1] <= le) ++lo;
    return lo;
}

constexpr int64_t kOneQ63 = INT64_MAX;

// Cell and fraction (Q63) of v on a uniform log10 axis, clamped to it (zero, negative, NaN: its lower end).
__device__ __forceinline__ void cell_q(double v, const FixedAxis& ax, const FixedTables& ft, int* i, int64_t* t) {
    int64_t z = log2_q52(v, ft) - ax.lo;
    z = z < 0 ? 0 : (z > ax.span ? ax.span : z);
    const uint64_t p = __umul64hi((uint64_t)z << ax.zs, ax.a);
    const int c = (int)(p >> ax.fb);
    const bool top = c > ax.n - 2;
    *i = top ? ax.n - 2 : c;
    *t = top ? kOneQ63 : (int64_t)((p << (64 - ax.fb)) >> 1);
}

// The same on a uniform linear axis: the coordinate in FP64, split by its bits.
__device__ __forceinline__ void cell_lin_q(double v, const Axis& ax, int* i, int64_t* t) {
    const uint64_t u = word_of((v - ax.lo) * ax.inv_d);
    const int e = (int)(u >> 52) - 1023;   // >= 1025 for a set sign bit
    const uint64_t m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 11;   // mantissa as Q63
    *i = 0;
    *t = 0;
    if (u > 0x7ff0000000000000ull) return;   // below the axis or NaN: its lower end
    if (e < 0) {
        if (e >= -62) *t = (int64_t)(m >> -e);
        return;
    }
    const int c = e > 30 ? INT32_MAX : (int)(m >> (63 - e));
    if (c > ax.n - 2) { *i = ax.n - 2; *t = kOneQ63; return; }
    *i = c;
    *t = (int64_t)(((m << e) << 1) >> 1);
}

__global__ void __launch_bounds__(kBuckets) opacity_interp_fixed_kernel(const DevGrid g, const DevTables tb, const InterpTables fx,
                                                                   int which, int species, long long p,
                                                                   const double* __restrict__ rho,
                                                                   const double* __restrict__ T,
                                                                   const double* __restrict__ Ye,
                                                                   const double* __restrict__ E,
                                                                   double* __restrict__ out) {
    __shared__ FixedTables ft;
    __shared__ int64_t lne[kMaxNe];
    __shared__ uint64_t rec[kMaxNe];
    __shared__ int sh[kMaxNe];
    __shared__ unsigned char lut[kBuckets];
    const int NE = g.ne;
    for (int k = threadIdx.x; k < (int)(sizeof(FixedTables) / 4); k += blockDim.x)
        reinterpret_cast<uint32_t*>(&ft)[k] = reinterpret_cast<const uint32_t*>(fx.ft)[k];
    for (int q = threadIdx.x; q < NE; q += blockDim.x) {
        lne[q] = fx.lne[q];
        rec[q] = fx.rec[q];
        sh[q] = fx.sh[q];
    }
    __syncthreads();
    // buckets of 2^shift of the Q52 logarithm
    const int64_t lo_e = lne[0], hi_e = lne[NE - 1];
    const int shift = max(0, 56 - (int)__clzll(hi_e - lo_e));   // (hi_e - lo_e) >> shift < kBuckets
    lut[threadIdx.x] = (unsigned char)cell_by_bisection(lne, NE, lo_e + ((int64_t)threadIdx.x - 1) * (int64_t(1) << shift));
    __syncthreads();
    const ulonglong2* __restrict__ tab = which == 0 ? fx.quads[0] : fx.quads[1];
    const long long nrc = tb.rho.n - 1, nec = NE - 1;
    const long long dT = nrc * nec, dY = (long long)tb.t.n * dT;
    const long long sp0 = (long long)species * tb.ye.n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < p; i += (long long)gridDim.x * blockDim.x) {
        int ir, it, iy;
        int64_t tr, tt, ty;
        cell_q(rho[i], fx.rho, ft, &ir, &tr);
        cell_q(T[i], fx.t, ft, &it, &tt);
        cell_lin_q(Ye[i], tb.ye, &iy, &ty);
        int64_t le = log2_q52(E[i], ft);
        le = le < lo_e ? lo_e : (le > hi_e ? hi_e : le);
        const int lo = cell_from(lne, NE, le, (int)lut[(le - lo_e) >> shift]);
        const long long base = (((sp0 + iy) * tb.t.n + it) * nrc + ir) * nec + lo;
        if (!NMC_IN_BOUNDS(g.dbg, base, fx.n_quad, kDbgEmabIso) ||
            !NMC_IN_BOUNDS(g.dbg, base + dT + dY, fx.n_quad, kDbgEmabIso))
            continue;
        ulonglong2 c[4][2];   // the (T, Ye) corners k = cb + 2 cc of the (rho, E) cell
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const ulonglong2* cp = tab + 2 * (base + (k & 1) * dT + (k >> 1) * dY);
            c[k][0] = __ldg(cp);
            c[k][1] = __ldg(cp + 1);
        }
        const uint64_t te62 = __umul64hi((uint64_t)(le - lne[lo]) << sh[lo], rec[lo]);
        const int64_t te = te62 >> 62 ? kOneQ63 : (int64_t)(te62 << 1);
        int64_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            v[k] = lerp_q(lerp_q((int64_t)c[k][0].x, (int64_t)c[k][0].y, te), lerp_q((int64_t)c[k][1].x, (int64_t)c[k][1].y, te), tr);
        out[i] = exp_q53(lerp_q(lerp_q(v[0], v[1], tt), lerp_q(v[2], v[3], tt), ty), ft);
    }
}

// The ln table [ns][nye][nt][nrho][ne] as Q53 cells (InterpTables).
__global__ void fixed_quads_kernel(const double* __restrict__ tab, long long nrows, int nr, int ne, ulonglong2* __restrict__ out) {
    const long long nrc = nr - 1, nec = ne - 1, total = nrows * nrc * nec;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long row = i / (nrc * nec), ir = (i / nec) % nrc, e = i % nec;
        const double* p0 = tab + (row * nr + ir) * ne + e;
        const double kQ = 9007199254740992.0;   // 2^53
        out[2 * i] = make_ulonglong2((unsigned long long)__double2ll_rn(p0[0] * kQ), (unsigned long long)__double2ll_rn(p0[1] * kQ));
        out[2 * i + 1] = make_ulonglong2((unsigned long long)__double2ll_rn(p0[ne] * kQ),
                                         (unsigned long long)__double2ll_rn(p0[ne + 1] * kQ));
    }
}

const FixedTables kFixedTables = {{NMC_LOG_L}, {NMC_EXP_T}, {NMC_LOG_C}};

// log10 axis [lo, hi] of n points; false when its constants do not fit
bool fixed_axis(double lo, double hi, int n, FixedAxis* ax) {
    if (!(lo >= -150.0 && hi <= 150.0) || n > (1 << 15)) return false;
    // log2(10) and log10(2) as double-doubles; products and the quotient to ~100 bits
    const double l2h = 3.321928094887362, l2l = 1.661617516973592e-16;
    const double lgh = 0.30102999566398120, lgl = -2.8037281277851704e-18;
    auto q52 = [&](double l) {
        const double p = l * l2h, e = std::fma(l, l2h, -p) + l * l2l;
        return (int64_t)std::llrint(p * 4503599627370496.0) + (int64_t)std::llrint(e * 4503599627370496.0);
    };
    ax->lo = q52(lo);
    ax->span = q52(hi) - ax->lo;
    ax->n = n;
    if (ax->span <= 0) return false;
    const double dh = hi - lo, bb = dh - hi, dl = (hi - (dh - bb)) - (lo + bb);
    const double nh = (n - 1) * lgh, nl = std::fma((double)(n - 1), lgh, -nh) + (n - 1) * lgl;
    const double q1 = nh / dh, q2 = (std::fma(-q1, dh, nh) + (nl - q1 * dl)) / dh;
    int ex = 0;
    std::frexp(q1, &ex);
    const int as = 64 - ex;   // a = q 2^as in [2^63, 2^64)
    ax->a = (uint64_t)std::ldexp(q1, as) + (uint64_t)(int64_t)std::llrint(std::ldexp(q2, as));
    ax->zs = __builtin_clzll((unsigned long long)ax->span) - 1;
    ax->fb = ax->zs + as - 12;
    return ax->fb >= 1 && ax->fb <= 63;
}

template <typename T>
int upload_fx(nmc_ctx* ctx, const T* host, size_t count, const T** dev) {
    void* p = nullptr;
    const int rc = device_alloc(ctx, count * sizeof(T), &p);
    if (rc != NMC_OK) return rc;
    const cudaError_t e = cudaMemcpy(p, host, count * sizeof(T), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return set_error(ctx, NMC_ECUDA, std::string("cudaMemcpy: ") + cudaGetErrorString(e));
    *dev = static_cast<const T*>(p);
    return NMC_OK;
}

__device__ __forceinline__ void cell_f(float v, const Axis& ax, int* i, float* t) {
    float x = (v - (float)ax.lo) * (float)ax.inv_d;
    if (!(x >= 0.0f)) x = 0.0f;
    if (x > (float)(ax.n - 1)) x = (float)(ax.n - 1);
    int c = (int)floorf(x);
    if (c > ax.n - 2) c = ax.n - 2;
    *i = c;
    *t = x - (float)c;
}

// U points per thread and step, so that their loads are in flight together; kCells: see the file's head.
template <int U, bool kCells>
__global__ void __launch_bounds__(kBuckets) opacity_interp_mixed_kernel(const DevGrid g, const DevTables tb, int which,
                                                                        int species, long long p,
                                                                        const double* __restrict__ rho,
                                                                        const double* __restrict__ T,
                                                                        const double* __restrict__ Ye,
                                                                        const double* __restrict__ E,
                                                                        double* __restrict__ out) {
    __shared__ float lne[kMaxNe];
    __shared__ unsigned char lut[kBuckets];
    const int NE = g.ne;
    for (int q = threadIdx.x; q < NE; q += blockDim.x) lne[q] = (float)g.lneps[q];
    __syncthreads();
    const float lo_e = lne[0], hi_e = lne[NE - 1], per_bucket = (hi_e - lo_e) / kBuckets, scale = kBuckets / (hi_e - lo_e);
    lut[threadIdx.x] = (unsigned char)cell_by_bisection(lne, NE, lo_e + ((int)threadIdx.x - 1) * per_bucket);
    __syncthreads();
    const float4* __restrict__ tab = which == 0 ? tb.emab_q : tb.iso_q;
    const float* __restrict__ row = which == 0 ? tb.emab_f : tb.iso_f;
    const int nt = kCells ? tb.t.n - 1 : tb.t.n, nr = kCells ? tb.rho.n - 1 : tb.rho.n, ne = kCells ? NE - 1 : NE;
    const long long dT = (long long)nr * ne, dY = nt * dT, sp0 = (long long)species * tb.ye.n;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; i0 < p; i0 += U * step) {
        float fr[U], ft[U], fy[U], fe[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = i0 + u * step < p ? i0 + u * step : i0;
            fr[u] = narrow(rho[i]);
            ft[u] = narrow(T[i]);
            fy[u] = narrow(Ye[i]);
            fe[u] = narrow(E[i]);
        }
        float tr[U], tt[U], ty[U], te[U];
        float4 c[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int ir, it, iy;
            cell_f(log10f(fr[u]), tb.rho, &ir, &tr[u]);
            cell_f(log10f(ft[u]), tb.t, &it, &tt[u]);
            cell_f(fy[u], tb.ye, &iy, &ty[u]);
            float le = logf(fe[u]);
            if (!(le >= lo_e)) le = lo_e;
            if (le > hi_e) le = hi_e;
            const int b = (int)((le - lo_e) * scale);
            const int lo = cell_from(lne, NE, le, (int)lut[b < kBuckets ? b : kBuckets - 1]);
            te[u] = (le - lne[lo]) / (lne[lo + 1] - lne[lo]);
            // the (T, rho, E) cell's eight corners are one 32-byte sector; (T, Ye) corners k = cb + 2 cc
            const long long base = (((sp0 + iy) * nt + it) * nr + ir) * ne + lo;
            const bool ok = NMC_IN_BOUNDS(g.dbg, base, kCells ? tb.n_quad : tb.n_op, kDbgEmabIso) &&
                            NMC_IN_BOUNDS(g.dbg, base + dY + (kCells ? 0 : dT + ne + 1), kCells ? tb.n_quad : tb.n_op, kDbgEmabIso);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                c[u][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!ok) continue;
                if constexpr (kCells) {
                    c[u][k] = __ldg(tab + 2 * (base + (k >> 1) * dY) + (k & 1));
                } else {
                    const float* r0 = row + base + (k & 1) * dT + (k >> 1) * dY;
                    c[u][k] = make_float4(__ldg(r0), __ldg(r0 + ne), __ldg(r0 + 1), __ldg(r0 + ne + 1));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float c0 = c[u][0].x;
            float v = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float wk = ((k & 1) ? tt[u] : 1.0f - tt[u]) * ((k >> 1) ? ty[u] : 1.0f - ty[u]);
                // rho_i and rho_i+1, each linear in ln E between the two energy nodes
                const float a0 = fmaf(te[u], c[u][k].z - c[u][k].x, c[u][k].x - c0);
                const float a1 = fmaf(te[u], c[u][k].w - c[u][k].y, c[u][k].y - c0);
                v = fmaf(wk, fmaf(tr[u], a1 - a0, a0), v);
            }
            if (i0 + u * step < p) out[i0 + u * step] = widen(expf(c0 + v));
        }
    }
}

// The FP32 ln table [ns][nye][nt][nrho][ne] regrouped per (T, rho, E) cell (DevTables::emab_q).
__global__ void f32_cells_kernel(const float* __restrict__ tab, long long nsy, int nt, int nr, int ne, float4* __restrict__ out) {
    const long long nrc = nr - 1, nec = ne - 1, ntc = nt - 1, total = nsy * ntc * nrc * nec;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long e = i % nec, ir = (i / nec) % nrc, it = (i / (nec * nrc)) % ntc, sy = i / (nec * nrc * ntc);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float* r0 = tab + ((sy * nt + it + k) * nr + ir) * ne + e;
            out[2 * i + k] = make_float4(r0[0], r0[ne], r0[1], r0[ne + 1]);
        }
    }
}

}  // namespace

int build_f32_cells(nmc_ctx* ctx) {
    DevTables& t = ctx->tb;
    const long long nsy = (long long)ctx->ns * t.ye.n;
    t.emab_q = t.iso_q = nullptr;
    t.n_quad = nsy * (t.t.n - 1) * (t.rho.n - 1) * (ctx->ne - 1);
    const size_t cells = (size_t)t.n_quad * 2;   // of one table, in float4
    void* p = nullptr;
    if (spare_alloc(ctx, 2 * cells * sizeof(float4), &p) != NMC_OK) return NMC_OK;
    float4* const q[2] = {static_cast<float4*>(p), static_cast<float4*>(p) + cells};
    for (int w = 0; w < 2; ++w)
        f32_cells_kernel<<<ctx->num_sms * 8, 256>>>(w == 0 ? t.emab_f : t.iso_f, nsy, t.t.n, t.rho.n, ctx->ne, q[w]);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);   // the fill's stream: others may be at work
    if (e != cudaSuccess) return set_error(ctx, NMC_ECUDA, std::string("FP32 cells: ") + cudaGetErrorString(e));
    t.emab_q = q[0];
    t.iso_q = q[1];
    return NMC_OK;
}

cudaError_t preload_interp() {
    cudaFuncAttributes fa;
    for (const void* k : {(const void*)opacity_interp_kernel, (const void*)opacity_interp_fixed_kernel,
                          (const void*)opacity_interp_mixed_kernel<1, true>,
                          (const void*)opacity_interp_mixed_kernel<2, true>,
                          (const void*)opacity_interp_mixed_kernel<1, false>}) {
        const cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int build_interp_tables(nmc_ctx* ctx, const nmc_tables* tb) {
    InterpTables& fx = ctx->fx;
    fx.quads[0] = fx.quads[1] = nullptr;
    const size_t n_op = (size_t)ctx->tb.n_op;
    for (const double* t : {tb->emab, tb->iso})
        for (size_t i = 0; i < n_op; ++i)
            if (!(std::fabs(t[i]) <= kFixedMax)) return NMC_OK;
    if (!fixed_axis(tb->lrho_min, tb->lrho_max, tb->n_rho, &fx.rho) || !fixed_axis(tb->lt_min, tb->lt_max, tb->n_t, &fx.t))
        return NMC_OK;
    const int ne = ctx->ne;
    std::vector<int64_t> lne(ne);
    std::vector<uint64_t> rec(ne, 0);
    std::vector<int> sh(ne, 0);
    for (int q = 0; q < ne; ++q) lne[q] = log2_q52(ctx->eps[q], kFixedTables);
    for (int q = 0; q + 1 < ne; ++q) {
        const int64_t d = lne[q + 1] - lne[q];
        if (d <= 0) return NMC_OK;
        sh[q] = __builtin_clzll((unsigned long long)d) - 1;
        const unsigned __int128 r = ((unsigned __int128)1 << 126) / ((unsigned __int128)d << sh[q]);   // den in [2^62, 2^63)
        rec[q] = r >> 64 ? UINT64_MAX : (uint64_t)r;
    }
    int rc = upload_fx(ctx, &kFixedTables, 1, &fx.ft);
    if (rc == NMC_OK) rc = upload_fx(ctx, lne.data(), lne.size(), &fx.lne);
    if (rc == NMC_OK) rc = upload_fx(ctx, rec.data(), rec.size(), &fx.rec);
    if (rc == NMC_OK) rc = upload_fx(ctx, sh.data(), sh.size(), &fx.sh);
    if (rc != NMC_OK) return rc == NMC_ENOMEM ? NMC_OK : rc;   // too little memory: the FP64 form serves
    const long long nrows = (long long)ctx->ns * tb->n_ye * tb->n_t;
    const size_t cells = (size_t)nrows * (tb->n_rho - 1) * (ne - 1) * 2;   // of one table, in ulonglong2
    void* p = nullptr;
    if (spare_alloc(ctx, 2 * cells * sizeof(ulonglong2), &p) != NMC_OK) return NMC_OK;
    ulonglong2* const q[2] = {static_cast<ulonglong2*>(p), static_cast<ulonglong2*>(p) + cells};
    for (int w = 0; w < 2; ++w)
        fixed_quads_kernel<<<ctx->num_sms * 8, 256>>>(w == 0 ? ctx->tb.emab : ctx->tb.iso, nrows, tb->n_rho, ne, q[w]);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);   // the fill's stream: others may be at work
    if (e != cudaSuccess) return set_error(ctx, NMC_ECUDA, std::string("fixed-point tables: ") + cudaGetErrorString(e));
    fx.n_quad = nrows * (tb->n_rho - 1) * (ne - 1);
    fx.quads[0] = q[0];
    fx.quads[1] = q[1];
    return NMC_OK;
}

int launch_opacity_interp_mixed(nmc_ctx* ctx, int which, int species, long long p, const double* rho,
                                const double* T, const double* Ye, const double* E, double* out,
                                cudaStream_t stream) {
    const int threads = kBuckets;
    long long blocks = (p + threads - 1) / threads;
    const long long cap = (long long)ctx->num_sms * 8;
    // two points a thread once every SM has its blocks; below that one, so that the points spread over the SMs
    const bool cells = ctx->tb.emab_q != nullptr;
    auto kern = !cells ? opacity_interp_mixed_kernel<1, false>
                       : (blocks >= 2 * cap ? opacity_interp_mixed_kernel<2, true> : opacity_interp_mixed_kernel<1, true>);
    kern<<<(unsigned)(blocks > cap ? cap : blocks), threads, 0, stream>>>(ctx->g, ctx->tb, which, species, p, rho, T, Ye, E, out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_error(ctx, NMC_ECUDA, std::string("opacity_interp_mixed launch: ") + cudaGetErrorString(e));
    return NMC_OK;
}

int launch_opacity_interp(nmc_ctx* ctx, int which, int species, long long p, const double* rho,
                          const double* T, const double* Ye, const double* E, double* out,
                          cudaStream_t stream) {
    const int threads = kBuckets;
    long long blocks = (p + threads - 1) / threads;
    const long long cap = (long long)ctx->num_sms * 8;
    if (blocks > cap) blocks = cap;
    if (ctx->fx.quads[0])
        opacity_interp_fixed_kernel<<<(unsigned)blocks, threads, 0, stream>>>(ctx->g, ctx->tb, ctx->fx, which, species, p, rho, T,
                                                                              Ye, E, out);
    else
        opacity_interp_kernel<<<(unsigned)blocks, threads, 0, stream>>>(ctx->g, ctx->tb, which, species, p, rho, T, Ye, E, out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(ctx, NMC_ECUDA, std::string("opacity_interp launch: ") + cudaGetErrorString(e));
    return NMC_OK;
}

}  // namespace nmc
