// Observables and data movement of liblbem:
//   * the FP64 near-to-far-field projection (Sec. 2.4, Eqs. 7-10 in the
//     far-field limit) and the angular intensity |S|^2 (Sec. 2.3, Eqs. 5-6);
//   * the field-energy monitor (Sec. 3.2: steady state is checked by the total
//     field energy) with its non-finite check;
//   * fields of the stored state, permittivity upload, population pack/unpack.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "step_cell.cuh"

namespace lbem {
namespace {

template <class S> __device__ __forceinline__ float ldv(const S *p);
template <> __device__ __forceinline__ float ldv<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float ldv<__half>(const __half *p) { return __half2float(*p); }
template <> __device__ __forceinline__ float ldv<__nv_bfloat16>(const __nv_bfloat16 *p) {
    return __bfloat162float(*p);
}
template <class S> __device__ __forceinline__ void stv(S *p, float v);
template <> __device__ __forceinline__ void stv<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void stv<__half>(__half *p, float v) { *p = __float2half_rn(v); }
template <> __device__ __forceinline__ void stv<__nv_bfloat16>(__nv_bfloat16 *p, float v) {
    *p = __float2bfloat16_rn(v);
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------------ far field
constexpr int kFFThreads = 256;
constexpr int kFFTableMax = 4480;   // phase entries held in shared memory (70 KB)
constexpr int kFFStaticMax = 1536;  // bytes of static shared memory of far_field_columns, at most (1152 in 3D)

// How a block of far_field_columns gets its phases exp(j k r_a (p_a - c_a)):
// evaluated at each use; as products of a coarse entry (every F-th coordinate)
// and a fine one (the F offsets), tabulated per block; or from a table of
// every coordinate of the box, filled with those products.  F = 2^fine_log2 gives
// the fewest entries.
enum FFPhase { FF_DIRECT = 0, FF_FACTORED = 1, FF_TABLE = 2 };

__host__ __device__ inline int ff_entries(int n, int lg) { return (1 << lg) + ((n + (1 << lg) - 1) >> lg); }
inline int ff_factored_entries(int mode, const FaceGeom &g, int lg)
{
    int e = 0;
    for (int ax = 0; ax < (mode == 2 ? 3 : 2); ++ax) e += ff_entries(g.hi[ax] - g.lo[ax] + 1, lg);
    return e;
}

// The outputs a mode has among N_xyz, L_xyz (Re, Im): EZ N_z, L_x, L_y; HZ N_x,
// N_y, L_z; 3D all twelve.  Output i of a mode's list, and an output's place.
template <int MODE> __host__ __device__ constexpr int ff_outs() { return MODE == 2 ? 12 : 6; }
template <int MODE> __host__ __device__ constexpr int ff_out(int i)
{
    return MODE == 2 ? i : (MODE == 0 ? 4 + i : (i < 4 ? i : 6 + i));
}

// Reduce-scatter of N = 8 or 16 values over the warp: each step a lane keeps the
// half of its values that its bit H selects and adds its partner's copy of that
// half; the steps that are left sum the one value.  Lane l then holds the warp's
// sum of value l / (32 / N).
template <int N> __device__ __forceinline__ double warp_scatter(double (&v)[N], int lane)
{
    int off = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h /= 2, off /= 2) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const double send = up ? v[j] : v[j + h];
            v[j] = (up ? v[j + h] : v[j]) + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    for (; off >= 1; off /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    return v[0];
}

// Stage 1: one block per (chunk of face columns, angle); writes 12 doubles
// (Re/Im of N_xyz, L_xyz).  The phase of face cell (iu, iv) factorises as
// t_u(iu) t_v(iv) t_w, and so does the trapezoidal weight, so one thread takes
// one face column (fixed iv; the threads of a warp read consecutive iv,
// coalesced) and sums the tangential phasors down the column with t_u(iu) w(iu)
// alone; the column factor t_v(iv) w(iv) t_w multiplies the four column sums
// once, and J = n x H, M = -n x E are formed from them.  Per (cell, angle) this
// is four complex multiply-adds.  Bound by the FP64 pipe (two operations a
// clock per SM), so what counts in 2D, where a column is one cell, is the FP64
// work beside the columns: the sincos of the phase entries, and the reduction
// over the block.  A table of every coordinate per block cost 16 blocks x 1970
// sincos an angle on a 1024^2 grid (0.60 ms for 181 angles); factored and with few
// blocks an angle the call took 0.127 ms; with the direction found by one warp,
// the faces' own factors kept, the fewest entries and a reduce-scatter of the
// mode's outputs alone it takes 0.100 (520^2 HZ: the kernel 48 -> 27 us, the call
// 92 -> 62).  A 4000^2 box, too long for that table, evaluated the phase of every
// (cell, angle): 0.97 -> 0.228 -> 0.182 ms.
template <int MODE, int PH>
__global__ void __launch_bounds__(kFFThreads) far_field_columns(const FarFieldArgs a)
{
    extern __shared__ double2 ff_tab[];
    constexpr int AXES = MODE == 2 ? 3 : 2;
    chain_release();
    const int ang = blockIdx.y;
    // the direction, by one warp (odd lanes take phi)
    __shared__ double rh[3];
    if (threadIdx.x < 32) {
        const bool odd = MODE == 2 && (threadIdx.x & 1);
        double sn, cs;
        sincos(odd ? a.phi[ang] : a.theta[ang], &sn, &cs);
        const double sp = __shfl_sync(0xffffffffu, sn, 1), cp = __shfl_sync(0xffffffffu, cs, 1);
        if (threadIdx.x == 0) {
            rh[0] = MODE == 2 ? sn * cp : cs;
            rh[1] = MODE == 2 ? sn * sp : sn;
            rh[2] = MODE == 2 ? cs : 0.0;
        }
    }
    __syncthreads();
    const int n3[3] = {a.g.hi[0] - a.g.lo[0] + 1, a.g.hi[1] - a.g.lo[1] + 1, a.g.hi[2] - a.g.lo[2] + 1};
    // factored entries of axis ax: the F fine ones at foff, then the coarse ones
    const int lg = a.fine_log2, fine = 1 << lg;
    const int foff[3] = {0, ff_entries(n3[0], lg), ff_entries(n3[0], lg) + ff_entries(n3[1], lg)};
    const int nfac = foff[2] + (AXES == 3 ? ff_entries(n3[2], lg) : 0);
    const int toff[3] = {nfac, nfac + n3[0], nfac + n3[0] + n3[1]};
    auto cmul = [](double2 p, double2 q) { return make_double2(p.x * q.x - p.y * q.y, p.x * q.y + p.y * q.x); };
    auto factored = [&](int ax, int e) {
        return cmul(ff_tab[foff[ax] + fine + (e >> lg)], ff_tab[foff[ax] + (e & (fine - 1))]);
    };
    auto phase = [&](int ax, int e) {
        if constexpr (PH == FF_TABLE) return ff_tab[toff[ax] + e];
        if constexpr (PH == FF_FACTORED) return factored(ax, e);
        double sp, cp;
        sincos(a.k * rh[ax] * (a.g.lo[ax] + e - a.center[ax]), &sp, &cp);
        return make_double2(cp, sp);
    };
    if constexpr (PH != FF_DIRECT) {
        for (int e = threadIdx.x; e < nfac; e += blockDim.x) {
            const int ax = e < foff[1] ? 0 : (AXES == 2 || e < foff[2] ? 1 : 2);
            const int i = e - foff[ax];
            const double pos = i < fine ? (double)i : a.g.lo[ax] + (double)(i - fine) * fine - a.center[ax];
            double sp, cp;
            sincos(a.k * rh[ax] * pos, &sp, &cp);
            ff_tab[e] = make_double2(cp, sp);
        }
        __syncthreads();
    }
    if constexpr (PH == FF_TABLE) {
        for (int e = threadIdx.x; e < n3[0] + n3[1] + n3[2]; e += blockDim.x) {
            const int ax = e < n3[0] ? 0 : (e < n3[0] + n3[1] ? 1 : 2);
            ff_tab[nfac + e] = factored(ax, e - (toff[ax] - nfac));
        }
        __syncthreads();
    }
    // the faces' own factors t_w, times the outward normal's sign
    __shared__ double2 tw[kMaxFaces];
    if (threadIdx.x < a.g.nfaces) {
        const int f = threadIdx.x, ax = a.g.axis[f];
        double2 p = phase(ax, a.g.side[f] ? n3[ax] - 1 : 0);
        if (!a.g.side[f]) p = make_double2(-p.x, -p.y);
        tw[f] = p;
    }
    __syncthreads();

    int ncols = 0;
    for (int f = 0; f < a.g.nfaces; ++f) ncols += a.g.nv[f];
    double acc[12];
#pragma unroll
    for (int m = 0; m < 12; ++m) acc[m] = 0.0;

    // the columns of one face at a time, so that the components are compile-time
    auto column = [&](auto axis, int f, int iv) {
        constexpr int ax = decltype(axis)::value;
        constexpr int ua = ax == 2 ? 1 : 2, va = ax == 0 ? 1 : 0;
        constexpr int b1 = (ax + 1) % 3, b2 = (ax + 2) % 3;
        constexpr int slot[4] = {slot_H(MODE, b1), slot_H(MODE, b2), slot_E(MODE, b1), slot_E(MODE, b2)};
        const int nu = a.g.nu[f], nv = a.g.nv[f];
        const long long plane = (long long)nu * nv;
        const double *base = a.dft + a.g.off[f] + iv;
        // column sums of t_u w_u X for X = H_b1, H_b2, E_b1, E_b2 (re, im)
        double sr[4] = {0, 0, 0, 0}, si[4] = {0, 0, 0, 0};
        if constexpr (MODE != 2) {  // one cell a column, t_u = 1
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (slot[q] >= 0) {
                    sr[q] = base[(2 * slot[q]) * plane];
                    si[q] = base[(2 * slot[q] + 1) * plane];
                }
        } else {
            for (int iu = 0; iu < nu; ++iu) {
                double2 p = phase(ua, iu);
                if (nu > 1 && (iu == 0 || iu == nu - 1)) {
                    p.x *= 0.5;
                    p.y *= 0.5;
                }
                const double *c = base + (long long)iu * nv;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double xr = c[(2 * slot[q]) * plane], xi = c[(2 * slot[q] + 1) * plane];
                    sr[q] = fma(p.x, xr, fma(-p.y, xi, sr[q]));
                    si[q] = fma(p.x, xi, fma(p.y, xr, si[q]));
                }
            }
        }
        // column factor t_v(iv) w_v(iv) t_w
        double2 cf = cmul(phase(va, iv), tw[f]);
        if (nv > 1 && (iv == 0 || iv == nv - 1)) {
            cf.x *= 0.5;
            cf.y *= 0.5;
        }
        // J_b1 = -sgn H_b2, J_b2 = sgn H_b1, M_b1 = sgn E_b2, M_b2 = -sgn E_b1
        auto add = [&](int m, double s, double xr, double xi) {
            acc[m] = fma(s * cf.x, xr, fma(-s * cf.y, xi, acc[m]));
            acc[m + 1] = fma(s * cf.x, xi, fma(s * cf.y, xr, acc[m + 1]));
        };
        if (slot[1] >= 0) add(2 * b1, -1.0, sr[1], si[1]);
        if (slot[0] >= 0) add(2 * b2, 1.0, sr[0], si[0]);
        if (slot[3] >= 0) add(6 + 2 * b1, 1.0, sr[3], si[3]);
        if (slot[2] >= 0) add(6 + 2 * b2, -1.0, sr[2], si[2]);
    };
    for (int col = blockIdx.x * kFFThreads + threadIdx.x; col < ncols; col += a.chunks * kFFThreads) {
        int f = 0, iv = col;
        while (iv >= a.g.nv[f]) iv -= a.g.nv[f++];
        const int ax = a.g.axis[f];
        if (ax == 0) column(std::integral_constant<int, 0>(), f, iv);
        else if (ax == 1) column(std::integral_constant<int, 1>(), f, iv);
        else if (MODE == 2) column(std::integral_constant<int, 2>(), f, iv);
    }

    constexpr int NO = ff_outs<MODE>(), N = MODE == 2 ? 16 : 8;
    __shared__ double red[kFFThreads / 32][N];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i < NO ? acc[ff_out<MODE>(i < NO ? i : 0)] : 0.0;
    const double sum = warp_scatter(v, lane);
    if (lane % (32 / N) == 0) red[wid][lane / (32 / N)] = sum;
    __syncthreads();
    static_assert(sizeof rh + sizeof tw + sizeof red <= kFFStaticMax, "the shared-memory opt-in counts them");
    if (threadIdx.x < 12) {
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < NO; ++i)
            if (ff_out<MODE>(i) == threadIdx.x)
                for (int wi = 0; wi < kFFThreads / 32; ++wi) s += red[wi][i];
        a.partial[((long long)ang * a.chunks + blockIdx.x) * 12 + threadIdx.x] = s;
    }
}

// Stage 2: fixed-order sum over chunks, then Eq. 5/6.  Twelve threads an angle
// sum one output each, then one lane an angle goes on.  FP64 again: a warp's
// instruction holds the pipe for 16 clocks however many lanes it has, so the
// angles are spread over the SMs and no lane repeats another's work (181 angles
// alone and cold: 10.4 us with 128 angles a block, 8.1 with eight).  What does not
// need the sums runs before the wait for them, beside the kernel that makes them.
constexpr int kFinAngles = 8;
__global__ void __launch_bounds__(12 * kFinAngles) far_field_finalize(const FarFieldArgs a)
{
    __shared__ double sums[kFinAngles * 12];
    const int ang0 = blockIdx.x * kFinAngles, ang = ang0 + threadIdx.x;
    const bool mine = threadIdx.x < kFinAngles && ang < a.n_ang;
    double ei = 0.0, st = 0.0, ct = 1.0, sp = 0.0, cp = 1.0;
    if (mine) {
        // |E_I|: incident-line E phasor along pol, mean over the two nodes around the centre
        const int nodes[2] = {a.center_i0, a.center_i1};
        for (int t = 0; t < 2 && a.ei_fixed <= 0.0; ++t) {
            double re = 0.0, im = 0.0;
            for (int c = 0; c < 3; ++c) {
                re += a.pol[c] * a.line_dft[(nodes[t] * 3 + c) * 2 + 0];
                im += a.pol[c] * a.line_dft[(nodes[t] * 3 + c) * 2 + 1];
            }
            ei += 0.5 * sqrt(re * re + im * im);
        }
        if (a.ei_fixed > 0.0) ei = a.ei_fixed;
        sincos(a.theta[ang], &st, &ct);
        if (a.mode == 2) sincos(a.phi[ang], &sp, &cp);
    }
    chain_wait();
    const int j = threadIdx.x / 12, m0 = threadIdx.x % 12;
    if (ang0 + j < a.n_ang) {
        const double *p = a.partial + (long long)(ang0 + j) * a.chunks * 12 + m0;
        double sum = 0.0;
#pragma unroll 8
        for (int c = 0; c < a.chunks; ++c) sum += p[c * 12];
        sums[threadIdx.x] = sum;
        if (a.amp) a.amp[(long long)ang0 * 12 + threadIdx.x] = sum;
    }
    __syncthreads();
    if (!mine) return;
    const double *v = sums + 12 * threadIdx.x;
    const double k = a.k;
    double s2;
    if (a.mode == 2) {
        const double tv[3] = {ct * cp, ct * sp, -st}, pv[3] = {-sp, cp, 0.0};
        double Nt[2] = {0, 0}, Np[2] = {0, 0}, Lt[2] = {0, 0}, Lp[2] = {0, 0};
        for (int c = 0; c < 3; ++c)
            for (int r = 0; r < 2; ++r) {
                Nt[r] += tv[c] * v[2 * c + r];
                Np[r] += pv[c] * v[2 * c + r];
                Lt[r] += tv[c] * v[6 + 2 * c + r];
                Lp[r] += pv[c] * v[6 + 2 * c + r];
            }
        const double a1r = Nt[0] + Lp[0], a1i = Nt[1] + Lp[1];
        const double a2r = Np[0] - Lt[0], a2i = Np[1] - Lt[1];
        s2 = k * k * k * k * (a1r * a1r + a1i * a1i + a2r * a2r + a2i * a2i) /
             (16.0 * M_PI * M_PI * ei * ei);
    } else {
        const double pv[3] = {-st, ct, 0.0};
        double Np[2] = {0, 0}, Lp[2] = {0, 0};
        for (int c = 0; c < 3; ++c)
            for (int r = 0; r < 2; ++r) {
                Np[r] += pv[c] * v[2 * c + r];
                Lp[r] += pv[c] * v[6 + 2 * c + r];
            }
        double ar, ai;
        if (a.mode == 0) { ar = v[4] - Lp[0]; ai = v[5] - Lp[1]; }      // N_z - L_phi
        else { ar = Np[0] + v[10]; ai = Np[1] + v[11]; }                // N_phi + L_z
        s2 = k * k * (ar * ar + ai * ai) / (8.0 * M_PI * ei * ei);
    }
    a.s2[ang] = s2;
}

// ------------------------------------------------------------ permittivity
// inv_eps == nullptr: only validate (eps_r finite and >= 1) into *bad.
__global__ void inv_eps_kernel(const float *eps, float *inv_eps, int nx, int ny, int nz, int nxp,
                               int *bad)
{
    const long long n = (long long)nx * ny * nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx);
        const long long r = i / nx;
        const float e = eps[i];
        if (inv_eps == nullptr) {
            if (!(e >= 1.0f) || !isfinite(e)) atomicOr(bad, 1);
        } else {
            inv_eps[r * nxp + x] = 1.0f / e;
        }
    }
}

// ------------------------------------------------------------ pack / unpack
// Incident population of plane q at cell (x, y, z) when it lies in the
// total-field box (where the stored value is the scattered part), else 0.
__device__ __forceinline__ float inc_at(const IncView &v, int q, int x, int y, int z)
{
    if (!v.on) return 0.f;
    if (x < v.tf_lo[0] || x > v.tf_hi[0] || y < v.tf_lo[1] || y > v.tf_hi[1] || z < v.tf_lo[2] ||
        z > v.tf_hi[2])
        return 0.f;
    if (v.on == 2) {
        // vacuum equilibrium (Eq. 2) of the analytic plane wave at the state's time
        const int i = plane_dir(v.mode, q), s = plane_slot(v.mode, q);
        if (i == 0) return 0.f;
        const int ne = mode_NE(v.mode);
        const int c = s < ne ? (v.mode == 0 ? 2 : s) : (v.mode == 1 ? 2 : s - ne);
        const float amp = (float)pw_amplitude(v.pw, x, y, z, v.t);
        const float E[3] = {amp * (float)v.pw.pol[0], amp * (float)v.pw.pol[1], amp * (float)v.pw.pol[2]};
        const float H[3] = {amp * (float)v.pw.kxp[0], amp * (float)v.pw.kxp[1], amp * (float)v.pw.kxp[2]};
        return s < ne ? (E[c] - cross_c(i, H, c)) * (1.0f / 6.0f) : (H[c] + cross_c(i, E, c)) * (1.0f / 6.0f);
    }
    const int s = v.axis == 0 ? x : (v.axis == 1 ? y : z);
    return v.line[(size_t)q * v.n + s];
}

__global__ void fill_kernel(float *p, long long n, float v)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        p[i] = v;
}

// Plane q of the stored populations: element base + w * cell (pop_index).
template <class S>
__global__ void pack_kernel(const S *f, int w, int q, float scale, float *out, int nx, int ny,
                            long long ncell, int nxp, IncView inc)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ncell;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx);
        const long long r = i / nx;
        const int y = (int)(r % ny), z = (int)(r / ny);
        out[i] = ldv<S>(f + w * (r * nxp + x)) * scale + inc_at(inc, q, x, y, z);
    }
}

template <class S>
__global__ void unpack_kernel(S *f, int w, int q, float inv_scale, const float *in, int nx, int ny,
                              long long ncell, int nxp, IncView inc)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ncell;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx);
        const long long r = i / nx;
        const int y = (int)(r % ny), z = (int)(r / ny);
        stv<S>(f + w * (r * nxp + x), (in[i] - inc_at(inc, q, x, y, z)) * inv_scale);
    }
}

// Convert the stored populations of the total-field box between the scattered
// part and the total (sign = +1: add the incident line, -1: remove it).
template <class S>
__global__ void add_incident_kernel(int mode, S *f, long long P, int Q, float scale, int nx, int ny,
                                    long long ncell, int nxp, IncView inc, float sign)
{
    const float inv = 1.0f / scale;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ncell;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx);
        const long long r = i / nx;
        const int y = (int)(r % ny), z = (int)(r / ny);
        for (int q = 0; q < Q; ++q) {
            const float add = inc_at(inc, q, x, y, z);
            if (add == 0.f) continue;
            S *p = f + pop_index(mode, (int)sizeof(S), P, q, r * nxp + x);
            stv<S>(p, (ldv<S>(p) * scale + sign * add) * inv);
        }
    }
}

// Total-field populations of n listed cells (x, y, z triplets): out[k][q].
template <int MODE, class S>
__global__ void probe_kernel(const S *f, float sc, long long P, int ny, int nxp, const int *xyz, int n,
                             IncView inc, float *out)
{
    constexpr int Q = Planes<MODE>::Q;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n * Q; j += gridDim.x * blockDim.x) {
        const int k = j / Q, q = j % Q;
        const int x = xyz[3 * k], y = xyz[3 * k + 1], z = xyz[3 * k + 2];
        const long long c = ((long long)z * ny + y) * nxp + x;
        out[j] = ldv<S>(f + pop_index(MODE, (int)sizeof(S), P, q, c)) * sc + inc_at(inc, q, x, y, z);
    }
}

template <int MODE, class S>
static cudaError_t probe_t(const void *f, float sc, long long P, int ny, int nxp, const int *xyz, int n,
                           const IncView &inc, float *out, cudaStream_t s)
{
    const int total = n * Planes<MODE>::Q;
    probe_kernel<MODE, S><<<(total + 255) / 256, 256, 0, s>>>((const S *)f, sc, P, ny, nxp, xyz, n, inc,
                                                              out);
    return cudaGetLastError();
}

// ------------------------------------------------------------ fields & energy
// D and B of the total field of the cell at (x, y, z), element c of a padded
// plane: the populations by vector loads of whole groups (a scalar load per
// population fetched every sector of a group two or four times, which with
// 64-bit divides held the old kernels at a tenth of the copy bandwidth), each
// population scaled and completed by its incident part before it is summed in
// direction order.  All populations are loaded before any incident part: with
// the two alternating per direction a cell took a load's latency seven times.
// The closed-form wave is evaluated once per cell.
template <int MODE, class S>
__device__ __forceinline__ void cell_DB(const S *f, float sc, long long P, int c, const IncView &inc, int x, int y,
                                        int z, float D[3], float B[3])
{
    using PL = Planes<MODE>;
    using M = Mode<MODE>;
    constexpr int NC = PL::NC, NE = PL::NE;
    float v[7 * NC];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const S *g = f + (long long)i * NC * P;
        float *w = v + i * NC;
        if constexpr (NC == 3) {
            Io<S>::ld2(g, c, w[0], w[1]);
            Io<S>::ld1(g + 2 * P, c, w[2]);
        } else if constexpr (sizeof(S) == 4) {
            Io<S>::ld2(g, c, w[0], w[1]);
            Io<S>::ld2(g + 2 * P, c, w[2], w[3]);
            Io<S>::ld2(g + 4 * P, c, w[4], w[5]);
        } else {
            Io<S>::ld4(g, c, w[0], w[1], w[2], w[3]);
            Io<S>::ld2(g + 4 * P, c, w[4], w[5]);
        }
    }
    const bool in = inc.on && in_box(x, y, z, inc.tf_lo, inc.tf_hi);
    if (in && inc.on == 1) {
        const float *l = inc.line + (inc.axis == 0 ? x : (inc.axis == 1 ? y : z));
        float add[7 * NC];
#pragma unroll
        for (int k = 0; k < 7 * NC; ++k) add[k] = __ldg(l + (size_t)slot_plane(MODE, k / NC, k % NC) * inc.n);
#pragma unroll
        for (int k = 0; k < 7 * NC; ++k) v[k] = v[k] * sc + add[k];
    } else if (in) {
        const float amp = (float)pw_amplitude(inc.pw, x, y, z, inc.t);
        float E0[3], H0[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            E0[k] = amp * (float)inc.pw.pol[k];
            H0[k] = amp * (float)inc.pw.kxp[k];
        }
#pragma unroll
        for (int k = 0; k < 7 * NC; ++k) {
            const int i = k / NC, s = k % NC, a = s < NE ? M::ec(s) : M::hc(s - NE);
            const float add = i == 0 ? 0.f
                                     : (s < NE ? E0[a] - cross_c(i, H0, a) : H0[a] + cross_c(i, E0, a)) * (1.0f / 6.0f);
            v[k] = v[k] * sc + add;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 7 * NC; ++k) v[k] *= sc;
    }
    D[0] = D[1] = D[2] = 0.f;
    B[0] = B[1] = B[2] = 0.f;
#pragma unroll
    for (int k = 0; k < 7 * NC; ++k) {
        const int s = k % NC;
        if (s < NE) D[M::ec(s)] += v[k];
        else B[M::hc(s - NE)] += v[k];
    }
}

constexpr int kEThreads = 256;

// E and H maps in one pass over the populations (components 0..2: E, 3..5: H;
// a null pointer is skipped).  Bound by HBM: the populations and 1/eps_r once,
// 4 B a component out.  One launch a component read the populations six times:
// 384^3 FP32 59.9 -> 1.59 ms, FP16 57.4 -> 1.31, 1024^2 EZ 0.575 -> 0.047.
struct FieldOut { float *p[6]; };
template <int MODE, class S>
__global__ void __launch_bounds__(kEThreads) fields_kernel(const S *f, const float *inv_eps, const float *inv_mu,
                                                           float sc, long long P, int nx, int ny, int nz, int nxp,
                                                           IncView inc, FieldOut out)
{
    const unsigned c = blockIdx.x * kEThreads + threadIdx.x;  // the padded plane has less than 2^31 cells
    if (c >= (unsigned)P) return;
    const unsigned r = c / (unsigned)nxp, x = c - r * (unsigned)nxp;
    if (x >= (unsigned)nx) return;
    const int z = (int)(r / (unsigned)ny), y = (int)(r - (unsigned)z * (unsigned)ny);
    float D[3], B[3];
    cell_DB<MODE, S>(f, sc, P, (int)c, inc, (int)x, y, z, D, B);
    const float ie = inv_eps[c], im = inv_mu ? inv_mu[c] : 1.0f;
    const long long i = (long long)r * nx + x;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (out.p[k]) out.p[k][i] = D[k] * ie;
        if (out.p[3 + k]) out.p[3 + k][i] = B[k] * im;
    }
}

// Field energy 1/2 sum (|D|^2 / eps + |B|^2 / mu), FP64 per block; HBM and the
// FP64 pipe (about 15 operations a cell) take about the same time in FP32
// storage.  384^3 FP32 15.8 -> 1.84 ms, FP16 14.3 -> 1.84, 1024^2 EZ 0.355 -> 0.073.
template <int MODE, class S>
__global__ void __launch_bounds__(kEThreads) energy_partial(const S *f, const float *inv_eps, const float *inv_mu,
                                                            float sc, long long P, int nx, int ny, int nxp,
                                                            IncView inc, double *partial)
{
    double acc = 0.0;
    for (long long cl = blockIdx.x * (long long)kEThreads + threadIdx.x; cl < P; cl += (long long)gridDim.x * kEThreads) {
        const unsigned c = (unsigned)cl;
        const unsigned r = c / (unsigned)nxp, x = c - r * (unsigned)nxp;
        if (x >= (unsigned)nx) continue;
        const int z = (int)(r / (unsigned)ny), y = (int)(r - (unsigned)z * (unsigned)ny);
        float D[3], B[3];
        cell_DB<MODE, S>(f, sc, P, (int)c, inc, (int)x, y, z, D, B);
        const double ie = inv_eps[c];
        double d = 0.0, b = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (in_e<MODE>(k)) d = fma((double)D[k], (double)D[k], d);
            if (in_h<MODE>(k)) b = fma((double)B[k], (double)B[k], b);
        }
        if (inv_mu) b *= (double)inv_mu[c];
        acc += fma(d, ie, b);
    }
    __shared__ double red[kEThreads / 32];
    const double v = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kEThreads / 32; ++w) s += red[w];
        partial[blockIdx.x] = s;
    }
}

// Half the sum of the block partials, in a fixed order, and beside it the
// kernel status word, so that one copy brings both back.  (One thread summing
// a few thousand partials took longer than the pass over a 2D grid.)
__global__ void __launch_bounds__(kEThreads) sum_partials(const double *partial, int n, const int *status, double *out)
{
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += kEThreads) acc += partial[i];
    __shared__ double red[kEThreads / 32];
    const double v = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kEThreads / 32; ++w) s += red[w];
        out[0] = 0.5 * s;
        out[1] = (double)*status;
    }
}

inline int grid_for(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    const long long cap = 32LL * std::max(1, sm_count());
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}


// ---------------------------------------------------------------------------
// 3D far field as an FP32 contraction.  With the phase factorised as above,
// the projection of face f is, per angle a and tangential component X,
//   sum_v t_v(a, v) t_w(a) sum_u t_u(a, u) w_u w_v X(u, v),
// a complex matrix product [angles x u] . [u x (v, X)] followed by a short
// contraction over v.  GB300's FP64 pipe runs at 1/64 of its FP32 rate, so
// the FP64 column kernel above spends ~17 ms on a 384^3 sphere's 543 angles.
// Here the products and the sums over at most uc face rows (and over the 64
// columns of a tile) are FP32, and everything above that (column tiles, row
// chunks, faces) is summed in FP64, in a fixed order.  Phases are evaluated in
// FP64 and rounded once; the phasors are rounded once to FP32.  A term then
// carries ~2^-23 relative error and a partial FP32 sum of n terms at most
// n 2^-24 of its absolute sum (n <= uc = 16..512 rows, or 64 columns).
constexpr int kF32Threads = 256;
constexpr int kF32Angles = 32;   // angles per block: 8 warps x 4
constexpr int kF32Cols = 64;     // face columns per tile: 32 lanes x 2
constexpr int kF32Rows = 16;     // face rows staged in shared memory per pass

// Phase tables tab32[e][a] = exp(j k r_ax(a) (p_e - c_ax)) for the box
// coordinates p_e along x, y, z (e in [0, n0 + n1 + n2)); zero for padded angles.
// A block fills 32 angles x 32 coordinates of one axis with products of 4 coarse
// and 8 fine phases an angle, formed from two phases by multiplication: FP64-bound,
// and a sincos and the direction's own sines per entry were ten times the work
// (the whole call, 543 angles: 384^3 0.600 -> 0.504 ms, 64^3 0.113 -> 0.088).
constexpr int kTabCoords = 32, kTabFine = 8;
__device__ __forceinline__ void ff32_tables(const FarFieldArgs &a, int block)
{
    __shared__ double2 fine[kTabFine + 1][32], coarse[kTabCoords / kTabFine][32];
    const int tiles = a.n_ang_pad / 32;
    const int ang0 = block % tiles * 32;
    int ax = 0, e0 = block / tiles * kTabCoords, toff = 0, n = a.g.hi[0] - a.g.lo[0] + 1;
    while (e0 >= n) {
        e0 -= (n + kTabCoords - 1) / kTabCoords * kTabCoords;
        toff += n;
        ++ax;
        n = a.g.hi[ax] - a.g.lo[ax] + 1;
    }
    auto cmul = [](double2 p, double2 q) { return make_double2(p.x * q.x - p.y * q.y, p.x * q.y + p.y * q.x); };
    const int j = threadIdx.x % 32, wid = threadIdx.x / 32, ang = ang0 + j;
    double2 first = make_double2(1.0, 0.0);
    if (wid < 2 && ang < a.n_ang) {   // the phase of one cell, and of the block's first coordinate
        const double th = a.theta[ang];
        const double r = ax == 2 ? cos(th) : sin(th) * (ax == 0 ? cos(a.phi[ang]) : sin(a.phi[ang]));
        sincos(a.k * r * (wid == 0 ? 1.0 : a.g.lo[ax] + (double)e0 - a.center[ax]), &first.y, &first.x);
    }
    if (wid == 0) {
        const double2 p2 = cmul(first, first), p4 = cmul(p2, p2);
        fine[0][j] = make_double2(1.0, 0.0);
        fine[1][j] = first;
        fine[2][j] = p2;
        fine[3][j] = cmul(p2, first);
        fine[4][j] = p4;
        fine[5][j] = cmul(p4, first);
        fine[6][j] = cmul(p4, p2);
        fine[7][j] = cmul(p4, cmul(p2, first));
        fine[8][j] = cmul(p4, p4);
    }
    __syncthreads();
    if (wid == 1) {
        const double2 p8 = fine[8][j], p16 = cmul(p8, p8);
        coarse[0][j] = first;
        coarse[1][j] = cmul(first, p8);
        coarse[2][j] = cmul(first, p16);
        coarse[3][j] = cmul(first, cmul(p16, p8));
    }
    __syncthreads();
    for (int i = wid; i < min(kTabCoords, n - e0); i += kF32Threads / 32) {
        const double2 p = cmul(coarse[i / kTabFine][j], fine[i % kTabFine][j]);
        a.tab32[(long long)(toff + e0 + i) * a.n_ang_pad + ang] =
            ang < a.n_ang ? make_float2((float)p.x, (float)p.y) : make_float2(0.f, 0.f);
    }
}

// Packed faces x32[f][u][q][v] = w_u w_v X_q(u, v) in FP32, q = H_b1, H_b2,
// E_b1, E_b2 (b1 = AX+1, b2 = AX+2 mod 3); zero in the padding.
__device__ __forceinline__ void ff32_pack(const FarFieldArgs &a, int block)
{
    const long long i = (long long)block * kF32Threads + threadIdx.x;
    if (i >= a.off32[a.g.nfaces]) return;
    int f = 0;
    while (i >= a.off32[f + 1]) ++f;
    const long long r = i - a.off32[f];
    const int nvp = a.nvp[f];
    int v;
    long long t;
    if (r < 0x7fffffffLL) {   // 32-bit division wherever it serves
        v = (int)((unsigned)r % (unsigned)nvp);
        t = (unsigned)r / (unsigned)nvp;
    } else {
        v = (int)(r % nvp);
        t = r / nvp;
    }
    const int q = (int)(t % 4), u = (int)(t / 4);
    const int nu = a.g.nu[f], nv = a.g.nv[f];
    float2 out = make_float2(0.f, 0.f);
    if (u < nu && v < nv) {
        const int ax = a.g.axis[f], b1 = (ax + 1) % 3, b2 = (ax + 2) % 3;
        const int slot = q == 0 ? slot_H(2, b1) : q == 1 ? slot_H(2, b2) : q == 2 ? slot_E(2, b1) : slot_E(2, b2);
        const long long plane = (long long)nu * nv;
        const double *c = a.dft + a.g.off[f] + (long long)u * nv + v;
        double w = 1.0;
        if (nu > 1 && (u == 0 || u == nu - 1)) w *= 0.5;
        if (nv > 1 && (v == 0 || v == nv - 1)) w *= 0.5;
        out = make_float2((float)(w * c[(2 * slot) * plane]), (float)(w * c[(2 * slot + 1) * plane]));
    }
    a.x32[i] = out;
}

// Both, in one launch: the first tab_blocks blocks take the tables.
__global__ void __launch_bounds__(kF32Threads) ff32_prepare(const FarFieldArgs a, int tab_blocks)
{
    chain_release();
    if ((int)blockIdx.x < tab_blocks) ff32_tables(a, blockIdx.x);
    else ff32_pack(a, blockIdx.x - tab_blocks);
}

__device__ __forceinline__ void cmac(float &sr, float &si, float2 p, float xr, float xi)
{
    sr = fmaf(p.x, xr, fmaf(-p.y, xi, sr));
    si = fmaf(p.x, xi, fmaf(p.y, xr, si));
}

// One step of a reduce-scatter over the warp: a lane keeps the half of its
// values selected by its bit H and adds the partner's copy of that half.
// After the steps 16, 8, 4, 2, 1, lane l holds the warp's sum of value l.
template <int H>
__device__ __forceinline__ void rs_stage(float (&o)[32], int lane)
{
    const bool up = (lane & H) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const float send = up ? o[i] : o[i + H];
        const float keep = up ? o[i + H] : o[i];
        o[i] = keep + __shfl_xor_sync(0xffffffffu, send, H);
    }
}

// One block per (tile of 32 angles, chunk of uc rows of one face).  Warp w
// owns angles 4w..4w+3 of the tile and lane l columns 2l, 2l+1 of each
// 64-column tile.  Per column tile: FP32 column sums over the chunk's rows,
// then the column factor, a reduce-scatter over the warp (lane l ends with
// value l of the warp's 4 angles x 8 outputs), and an FP64 add into shared
// memory.  Writes partial[angle][chunk][12].
__global__ void __launch_bounds__(kF32Threads, 2) far_field_f32(const FarFieldArgs a)
{
    extern __shared__ float4 ff_sm[];
    chain_release();
    chain_wait();
    float2 *At = reinterpret_cast<float2 *>(ff_sm);                  // [uc][32] row phases
    float4 *Xs = ff_sm + a.uc * (kF32Angles / 2);                    // [16 rows x 4 q][32] (2 columns)
    double *acc = reinterpret_cast<double *>(Xs + kF32Rows * 4 * 32);  // [32 angles][12]
    const int lane = threadIdx.x & 31, wg = threadIdx.x >> 5;
    const int ang0 = blockIdx.x * kF32Angles;
    const int ch = blockIdx.y;
    int f = 0;
    while (f + 1 < a.g.nfaces && ch >= a.chunk_start[f + 1]) ++f;
    const int u0 = (ch - a.chunk_start[f]) * a.uc;
    const int nu = a.g.nu[f], nv = a.g.nv[f], nvp = a.nvp[f];
    const int un = min(a.uc, a.nup[f] - u0);  // a multiple of kF32Rows
    const int ax = a.g.axis[f];
    const int ua = ax == 2 ? 1 : 2, va = ax == 0 ? 1 : 0;
    const int b1 = (ax + 1) % 3, b2 = (ax + 2) % 3;
    const int n0 = a.g.hi[0] - a.g.lo[0] + 1, n1 = a.g.hi[1] - a.g.lo[1] + 1;
    auto toff = [&](int axis) { return axis == 0 ? 0 : (axis == 1 ? n0 : n0 + n1); };
    const int eu = toff(ua), ev = toff(va);
    for (int i = threadIdx.x; i < un * kF32Angles; i += kF32Threads) {
        const int u = i / kF32Angles, j = i % kF32Angles;
        At[i] = u0 + u < nu ? a.tab32[(long long)(eu + u0 + u) * a.n_ang_pad + ang0 + j]
                            : make_float2(0.f, 0.f);
    }
    for (int i = threadIdx.x; i < kF32Angles * 12; i += kF32Threads) acc[i] = 0.0;
    const int ew = toff(ax) + (a.g.side[f] ? a.g.hi[ax] - a.g.lo[ax] : 0);
    const double sgn = a.g.side[f] ? 1.0 : -1.0;
    const float4 *X = reinterpret_cast<const float4 *>(a.x32 + a.off32[f]);
    const int nvq = nvp / 2;  // float4 (two columns) per row of one component
    // output slot of reduce-scatter value q of an angle: J_b1, J_b2, M_b1, M_b2 (re, im)
    const int qv = lane & 7, jv = lane >> 3;
    const int mslot = (qv < 4 ? 0 : 6) + 2 * ((qv & 2) ? b2 : b1) + (qv & 1);

    for (int c0 = 0; c0 < nvp; c0 += kF32Cols) {
        float sr[4][2][4], si[4][2][4];  // [angle][column][q]
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int q = 0; q < 4; ++q) sr[j][c][q] = si[j][c][q] = 0.f;
        for (int s0 = 0; s0 < un; s0 += kF32Rows) {
            __syncthreads();
            for (int i = threadIdx.x; i < kF32Rows * 4 * 32; i += kF32Threads) {
                const int row = i >> 5, l = i & 31;  // row = us * 4 + q
                Xs[i] = X[(long long)((u0 + s0) * 4 + row) * nvq + c0 / 2 + l];
            }
            __syncthreads();
#pragma unroll 2
            for (int us = 0; us < kF32Rows; ++us) {
                const float4 *pw = reinterpret_cast<const float4 *>(At + (s0 + us) * kF32Angles + 4 * wg);
                const float4 pa = pw[0], pb = pw[1];
                const float2 p[4] = {make_float2(pa.x, pa.y), make_float2(pa.z, pa.w),
                                     make_float2(pb.x, pb.y), make_float2(pb.z, pb.w)};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 x = Xs[(us * 4 + q) * 32 + lane];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        cmac(sr[j][0][q], si[j][0][q], p[j], x.x, x.y);
                        cmac(sr[j][1][q], si[j][1][q], p[j], x.z, x.w);
                    }
                }
            }
        }
        // column factor t_v t_w; J_b1 = -H_b2, J_b2 = H_b1, M_b1 = E_b2, M_b2 = -E_b1
        // (times the normal's sign, applied in FP64 below)
        float o[32];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long ang = ang0 + 4 * wg + j;
            const float2 tw = a.tab32[(long long)ew * a.n_ang_pad + ang];
#pragma unroll
            for (int q = 0; q < 8; ++q) o[8 * j + q] = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int v = c0 + 2 * lane + c;
                const float2 tv = v < nv ? a.tab32[(long long)(ev + v) * a.n_ang_pad + ang]
                                         : make_float2(0.f, 0.f);
                const float cr = tv.x * tw.x - tv.y * tw.y, ci = tv.x * tw.y + tv.y * tw.x;
                const float sg[4] = {1.f, -1.f, -1.f, 1.f};   // sign of q in its output
                const int oq[4] = {2, 0, 6, 4};               // H_b1 -> J_b2, H_b2 -> J_b1, E_b1 -> M_b2, E_b2 -> M_b1
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float xr = sg[q] * sr[j][c][q], xi = sg[q] * si[j][c][q];
                    o[8 * j + oq[q]] = fmaf(cr, xr, fmaf(-ci, xi, o[8 * j + oq[q]]));
                    o[8 * j + oq[q] + 1] = fmaf(cr, xi, fmaf(ci, xr, o[8 * j + oq[q] + 1]));
                }
            }
        }
        rs_stage<16>(o, lane);
        rs_stage<8>(o, lane);
        rs_stage<4>(o, lane);
        rs_stage<2>(o, lane);
        rs_stage<1>(o, lane);
        acc[(4 * wg + jv) * 12 + mslot] += sgn * (double)o[0];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kF32Angles * 12; i += kF32Threads) {
        const int j = i / 12, m = i % 12;
        if (ang0 + j < a.n_ang) a.partial[((long long)(ang0 + j) * a.chunks + ch) * 12 + m] = acc[i];
    }
}

}  // namespace

static cudaError_t launch_finalize(const FarFieldArgs &a, cudaStream_t s)
{
    return launch_chained(true, far_field_finalize, (a.n_ang + kFinAngles - 1) / kFinAngles, 12 * kFinAngles, 0, s, a);
}

static size_t ff32_smem(int uc)
{
    return (size_t)uc * kF32Angles * sizeof(float2) + (size_t)kF32Rows * 4 * 32 * sizeof(float4) +
           (size_t)kF32Angles * 12 * sizeof(double);
}

// The 3D projection through far_field_f32: phase tables, packed faces, the
// contraction and the FP64 finalisation.  The chunk height uc (a multiple of
// 16 rows) minimises waves x (uc + 8): fewer, taller chunks waste less per
// block but quantise the grid into more partial waves.
static cudaError_t launch_far_field_f32(FarFieldArgs a, cudaStream_t s, int *launches)
{
    if (a.n_ang <= 0) return cudaSuccess;
    long long off = 0;
    for (int f = 0; f < a.g.nfaces; ++f) {
        a.nup[f] = (a.g.nu[f] + kF32Rows - 1) / kF32Rows * kF32Rows;
        a.nvp[f] = (a.g.nv[f] + kF32Cols - 1) / kF32Cols * kF32Cols;
        a.off32[f] = off;
        off += (long long)a.nup[f] * 4 * a.nvp[f];
    }
    a.off32[a.g.nfaces] = off;
    a.n_ang_pad = (a.n_ang + kF32Angles - 1) / kF32Angles * kF32Angles;
    const int ne = (a.g.hi[0] - a.g.lo[0] + 1) + (a.g.hi[1] - a.g.lo[1] + 1) + (a.g.hi[2] - a.g.lo[2] + 1);
    if (off > a.x32_cap || (long long)ne * a.n_ang_pad > a.tab32_cap) return cudaErrorInvalidValue;
    // resident blocks per SM for each chunk height (shared memory grows with
    // uc), and the shared-memory opt-in: once per device
    constexpr int kMaxUc = 512;
    static std::mutex setup_mu;
    static bool ready_of[kMaxDevices];
    static int per_uc_of[kMaxDevices][kMaxUc / kF32Rows + 1];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const int sms = sm_count();
    if (sms < 1) return cudaErrorInvalidDevice;
    int per_uc[kMaxUc / kF32Rows + 1];
    {
        std::lock_guard<std::mutex> lock(setup_mu);
        if (!ready_of[dev]) {
            e = cudaFuncSetAttribute(far_field_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)ff32_smem(kMaxUc));
            for (int uc = kF32Rows; e == cudaSuccess && uc <= kMaxUc; uc += kF32Rows)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_uc_of[dev][uc / kF32Rows], far_field_f32,
                                                                   kF32Threads, ff32_smem(uc));
            if (e != cudaSuccess) return e;
            ready_of[dev] = true;
        }
        std::memcpy(per_uc, per_uc_of[dev], sizeof per_uc);
    }
    const int tiles = a.n_ang_pad / kF32Angles;
    int best_uc = 0;
    double best = 0.0;
    for (int uc = kF32Rows; uc <= kMaxUc; uc += kF32Rows) {
        int chunks = 0;
        for (int f = 0; f < a.g.nfaces; ++f) chunks += (a.nup[f] + uc - 1) / uc;
        const int per = per_uc[uc / kF32Rows];
        if (chunks > kMaxChunks || per < 1) continue;
        const long long blocks = (long long)tiles * chunks;
        const long long waves = (blocks + (long long)per * sms - 1) / ((long long)per * sms);
        const double t = (double)waves * (uc + 8);
        if (best_uc == 0 || t < best) {
            best = t;
            best_uc = uc;
        }
    }
    if (best_uc == 0) return cudaErrorInvalidValue;
    a.uc = best_uc;
    a.chunk_start[0] = 0;
    for (int f = 0; f < a.g.nfaces; ++f) a.chunk_start[f + 1] = a.chunk_start[f] + (a.nup[f] + a.uc - 1) / a.uc;
    a.chunks = a.chunk_start[a.g.nfaces];
    const size_t sm = ff32_smem(a.uc);
    long long tab_blocks = 0;
    for (int ax = 0; ax < 3; ++ax) tab_blocks += (a.g.hi[ax] - a.g.lo[ax] + kTabCoords) / kTabCoords;
    tab_blocks *= a.n_ang_pad / 32;
    const long long blocks = tab_blocks + (off + kF32Threads - 1) / kF32Threads;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    ff32_prepare<<<(unsigned)blocks, kF32Threads, 0, s>>>(a, (int)tab_blocks);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_chained(true, far_field_f32, dim3(tiles, a.chunks), kF32Threads, sm, s, a);
    if (e == cudaSuccess) e = launch_finalize(a, s);
    if (launches) *launches += 3;
    return e;
}

// The FP64 projection's partial sums (the caller finalises).  In 3D a column
// has many cells, so every coordinate's phase is tabulated where that fits; 2D
// boxes use each entry once and take the factored phases.
template <int MODE, int PH>
static cudaError_t far_field_columns_go(const FarFieldArgs &a, int entries, cudaStream_t s)
{
    const size_t smem = (size_t)entries * sizeof(double2);
    // static and dynamic shared memory together stay within 48 KB without the opt-in
    if (smem + kFFStaticMax > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(far_field_columns<MODE, PH>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kFFTableMax * (int)sizeof(double2));
        if (e != cudaSuccess) return e;
    }
    far_field_columns<MODE, PH><<<dim3(a.chunks, a.n_ang), kFFThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t far_field_columns_t(FarFieldArgs a, cudaStream_t s)
{
    a.fine_log2 = 3;
    for (int lg = 4; lg <= 8; ++lg)
        if (ff_factored_entries(MODE, a.g, lg) < ff_factored_entries(MODE, a.g, a.fine_log2)) a.fine_log2 = lg;
    const int fac = ff_factored_entries(MODE, a.g, a.fine_log2);
    if constexpr (MODE == 2) {
        int all = fac;
        for (int ax = 0; ax < 3; ++ax) all += a.g.hi[ax] - a.g.lo[ax] + 1;
        if (all <= kFFTableMax) return far_field_columns_go<MODE, FF_TABLE>(a, all, s);
    }
    if (fac <= kFFTableMax) return far_field_columns_go<MODE, FF_FACTORED>(a, fac, s);
    return far_field_columns_go<MODE, FF_DIRECT>(a, 0, s);
}

cudaError_t launch_far_field_partial(const FarFieldArgs &a, cudaStream_t s)
{
    switch (a.mode) {
    case 0: return far_field_columns_t<0>(a, s);
    case 1: return far_field_columns_t<1>(a, s);
    case 2: return far_field_columns_t<2>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

// Blocks an angle of the FP64 projection: in 2D about three blocks per SM in
// all (each block pays for its phase entries), in 3D one per 4096 face cells;
// at most one per kFFThreads columns.
int far_field_chunks(int mode, const FaceGeom &g, int n_ang, int most)
{
    long long cols = 0;
    for (int f = 0; f < g.nfaces; ++f) cols += g.nv[f];
    const long long per_cols = (cols + kFFThreads - 1) / kFFThreads;
    long long c = std::max((g.cell_start[g.nfaces] + 4095) / 4096, per_cols);
    if (mode != 2) c = std::min<long long>(per_cols, (3LL * std::max(1, sm_count()) + n_ang - 1) / std::max(1, n_ang));
    return (int)std::max<long long>(1, std::min<long long>(most, c));
}

cudaError_t launch_far_field(const FarFieldArgs &a, cudaStream_t s, int *launches)
{
    if (a.mode == 2 && a.x32 != nullptr) return launch_far_field_f32(a, s, launches);
    const cudaError_t e = launch_far_field_partial(a, s);
    if (e != cudaSuccess) return e;
    if (launches) *launches += 2;
    return launch_finalize(a, s);
}

cudaError_t launch_fill(float *p, long long n, float v, cudaStream_t s)
{
    fill_kernel<<<grid_for(n, 256), 256, 0, s>>>(p, n, v);
    return cudaGetLastError();
}

cudaError_t launch_inv_eps(const float *eps, float *inv_eps, int nx, int ny, int nz, int nxp,
                           int *bad_flag, cudaStream_t s)
{
    const long long n = (long long)nx * ny * nz;
    inv_eps_kernel<<<grid_for(n, 256), 256, 0, s>>>(eps, inv_eps, nx, ny, nz, nxp, bad_flag);
    return cudaGetLastError();
}

cudaError_t launch_pack(int mode, int storage, const void *f, long long P, int q, float scale,
                        float *out, int nx, int ny, int nz, int nxp, const IncView &inc, cudaStream_t s)
{
    const long long n = (long long)nx * ny * nz;
    const int g = grid_for(n, 256);
    const int eb = storage == 0 ? 4 : 2;
    const long long base = pop_index(mode, eb, P, q, 0);
    const int w = (int)(pop_index(mode, eb, P, q, 1) - base);
    if (storage == 0)
        pack_kernel<float><<<g, 256, 0, s>>>((const float *)f + base, w, q, scale, out, nx, ny, n, nxp, inc);
    else if (storage == 1)
        pack_kernel<__half><<<g, 256, 0, s>>>((const __half *)f + base, w, q, scale, out, nx, ny, n, nxp, inc);
    else
        pack_kernel<__nv_bfloat16><<<g, 256, 0, s>>>((const __nv_bfloat16 *)f + base, w, q, scale, out, nx,
                                                     ny, n, nxp, inc);
    return cudaGetLastError();
}

cudaError_t launch_unpack(int mode, int storage, void *f, long long P, int q, float inv_scale,
                          const float *in, int nx, int ny, int nz, int nxp, const IncView &inc,
                          cudaStream_t s)
{
    const long long n = (long long)nx * ny * nz;
    const int g = grid_for(n, 256);
    const int eb = storage == 0 ? 4 : 2;
    const long long base = pop_index(mode, eb, P, q, 0);
    const int w = (int)(pop_index(mode, eb, P, q, 1) - base);
    if (storage == 0)
        unpack_kernel<float><<<g, 256, 0, s>>>((float *)f + base, w, q, inv_scale, in, nx, ny, n, nxp, inc);
    else if (storage == 1)
        unpack_kernel<__half><<<g, 256, 0, s>>>((__half *)f + base, w, q, inv_scale, in, nx, ny, n, nxp, inc);
    else
        unpack_kernel<__nv_bfloat16><<<g, 256, 0, s>>>((__nv_bfloat16 *)f + base, w, q, inv_scale, in, nx,
                                                       ny, n, nxp, inc);
    return cudaGetLastError();
}

cudaError_t launch_add_incident(int mode, int storage, void *f, long long P, int Q, float scale,
                                int nx, int ny, int nz, int nxp, const IncView &inc, float sign,
                                cudaStream_t s)
{
    const long long n = (long long)nx * ny * nz;
    const int g = grid_for(n, 256);
    if (storage == 0)
        add_incident_kernel<float><<<g, 256, 0, s>>>(mode, (float *)f, P, Q, scale, nx, ny, n, nxp, inc, sign);
    else if (storage == 1)
        add_incident_kernel<__half><<<g, 256, 0, s>>>(mode, (__half *)f, P, Q, scale, nx, ny, n, nxp, inc, sign);
    else
        add_incident_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(mode, (__nv_bfloat16 *)f, P, Q, scale, nx, ny, n,
                                                             nxp, inc, sign);
    return cudaGetLastError();
}

template <int MODE, class S>
static cudaError_t fields_t(const void *f, const float *inv_eps, const float *inv_mu, float sc,
                            long long P, int nx, int ny, int nz, int nxp, const IncView &inc,
                            float *const out[6], cudaStream_t s)
{
    FieldOut o;
    std::memcpy(o.p, out, sizeof o.p);
    fields_kernel<MODE, S><<<(unsigned)((P + kEThreads - 1) / kEThreads), kEThreads, 0, s>>>(
        (const S *)f, inv_eps, inv_mu, sc, P, nx, ny, nz, nxp, inc, o);
    return cudaGetLastError();
}

template <int MODE, class S>
static cudaError_t energy_t(const void *f, const float *inv_eps, const float *inv_mu, float sc, long long P,
                            int nx, int ny, int nxp, const IncView &inc, double *partial,
                            int max_partial, const int *status, double *out, cudaStream_t s)
{
    const long long need = (P + kEThreads - 1) / kEThreads, cap = 8LL * std::max(1, sm_count());
    const int g = (int)std::min<long long>(std::min(need, cap), max_partial);
    energy_partial<MODE, S><<<g, kEThreads, 0, s>>>((const S *)f, inv_eps, inv_mu, sc, P, nx, ny, nxp, inc, partial);
    sum_partials<<<1, kEThreads, 0, s>>>(partial, g, status, out);
    return cudaGetLastError();
}

#define LBEM_DISPATCH(FN, ...)                                                   \
    switch (mode * 3 + storage) {                                                \
    case 0: return FN<0, float>(__VA_ARGS__);                                    \
    case 1: return FN<0, __half>(__VA_ARGS__);                                   \
    case 2: return FN<0, __nv_bfloat16>(__VA_ARGS__);                            \
    case 3: return FN<1, float>(__VA_ARGS__);                                    \
    case 4: return FN<1, __half>(__VA_ARGS__);                                   \
    case 5: return FN<1, __nv_bfloat16>(__VA_ARGS__);                            \
    case 6: return FN<2, float>(__VA_ARGS__);                                    \
    case 7: return FN<2, __half>(__VA_ARGS__);                                   \
    case 8: return FN<2, __nv_bfloat16>(__VA_ARGS__);                            \
    default: return cudaErrorInvalidValue;                                       \
    }

cudaError_t launch_fields(int mode, int storage, const void *f, const float *inv_eps, const float *inv_mu,
                          float scale, long long P, int nx, int ny, int nz, int nxp,
                          const IncView &inc, float *const out[6], cudaStream_t s)
{
    LBEM_DISPATCH(fields_t, f, inv_eps, inv_mu, scale, P, nx, ny, nz, nxp, inc, out, s)
}

cudaError_t launch_probe(int mode, int storage, const void *f, float scale, long long P, int ny, int nxp,
                         const int *xyz, int n, const IncView &inc, float *out, cudaStream_t s)
{
    LBEM_DISPATCH(probe_t, f, scale, P, ny, nxp, xyz, n, inc, out, s)
}

cudaError_t launch_energy(int mode, int storage, const void *f, const float *inv_eps, const float *inv_mu,
                          float scale, long long P, int nx, int ny, int nxp, const IncView &inc, double *partial,
                          int max_partial, const int *status, double *out, cudaStream_t s, int *launches)
{
    if (launches) *launches += 2;
    LBEM_DISPATCH(energy_t, f, inv_eps, inv_mu, scale, P, nx, ny, nxp, inc, partial, max_partial, status, out, s)
}

}  // namespace lbem
