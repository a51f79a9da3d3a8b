// Four lattice updates per pass in 2D (Eq. 1 of arXiv 2510.11042 applied four
// times, the boundary of Eq. 4 at every pull): temporal blocking in registers.
//
// A block owns a strip of 56 cells along x and marches along y through a chunk
// of rows.  A warp owns a row at a time, two neighbouring cells to a lane, and
// keeps the row's populations in registers while it takes them through the
// four levels; the block's sixteen warps hold sixteen consecutive rows.
//   * Rest and +-z populations never leave the registers (a 2D grid pulls +-z
//     from the cell itself).
//   * +-x pulls are warp shuffles, so the outermost cells of the 64 a warp
//     holds go stale one per level: the neighbouring strip's blocks recompute
//     four on each side.
//   * +-y groups go through shared memory to the warps of the rows above and
//     below.  Level l+1 of a row waits, on an mbarrier per row slot and level,
//     for level l of these two rows only; there is no block barrier in the march.
//     A chunk recomputes up to three rows on each side.
//   * The next row's level n is copied into shared memory (cp.async) while the
//     warp is at the row before.
// Level n is read from memory and level n+4 written once per four steps.  Passes
// of two or three steps take what a call of few steps asks for, on large grids
// (short_passes in api.cu): the same kernel with fewer levels and the same strips.
// (Strips of 60 cells, which two levels would allow, start off the sectors' ends:
// 2048^2 EZ FP16 51 -> 54 us a step, 250 x 8000 FP16 34 -> 38; 3000^2 gained 7 %.)
//
// Every sum, product and rounding is that of update_cell (step_cell.cuh), two
// cells to a packed FP32x2 instruction; 16-bit storage rounds the levels between
// to the storage type as a single step stores them.  So the populations are
// bitwise those of four single steps.
//
// Bound on large grids by HBM (4000^2 EZ FP32: 171 B a cell and pass at 0.88 of
// the copy bandwidth), on smaller ones by instruction issue (2.0 instructions a
// clock per SM, about 240 per row and level) and the rows' waits.  us a step,
// single step or two-step pass before -> now (in the DFT window):
//   520^2 HZ FP32 8.5 -> 4.7 (12.1 -> 5.0), 1024^2 EZ FP32 20.6 -> 12.6 (32.5 ->
//   13.7), 1000^2 HZ FP16 16.6 -> 11.0 (21.0 -> 12.9), 4000^2 EZ FP32 217 -> 118
//   (264 -> 120).
// Tried: one warp marching on its own with the levels in its registers (8 warps
// an SM: 520^2 6.8, 4000^2 143); a block barrier per row instead of the waits
// (8.3, 390); eight warps a block and two blocks an SM (5.2, 174).
#include <algorithm>
#include <cstring>
#include <mutex>

#include "march.cuh"

namespace lbem {
namespace {

__device__ __forceinline__ void stage3(float *p, long long n, float v0, float v1, float v2)
{
    p[0] = v0;
    p[n] = v1;
    p[2 * n] = v2;
}

// update_cell for a lane's two cells at (x, r) and (x + 1, r): f[3 i + s] over
// directions and slots, pulled populations in, post-collision ones out.  lev:
// the step of the pass (fields of time n + 1 + lev).
template <int MODE, bool MU, bool REC>
__device__ __forceinline__ void update2(const MarchArgs &a, P2 *f, int lev, const Cols &cx, const RowFacts &row,
                                        P2 ie2, P2 im2)
{
    using PL = Planes<MODE>;
    constexpr int NE = PL::NE;
    P2 m[3], F[3], T[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        m[s] = f[s];
#pragma unroll
        for (int i = 1; i < 7; ++i) m[s] = add2(m[s], f[3 * i + s]);
        F[s] = s < NE ? mul2(m[s], ie2) : (MU ? mul2(m[s], im2) : m[s]);
    }
    const int r = row.r;
    if constexpr (REC) {
        // total-field D of the pulled populations, for the adjoint
        if (row.mine) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int x = cx.x + c;
                if (x >= a.nx) continue;
                const bool in = a.tfsf && x >= a.tf_lo[0] && x <= a.tf_hi[0] && r >= a.tf_lo[1] && r <= a.tf_hi[1];
                const int sl = a.inc_axis == 0 ? x : r;
#pragma unroll
                for (int s = 0; s < NE; ++s) {
                    const float inc = in ? a.lm[lev][(size_t)s * a.n_line + sl] : 0.f;
                    a.rec[lev][(long long)s * a.P + (long long)r * a.nxp + x] = (c ? un(m[s]).y : un(m[s]).x) * a.scale + inc;
                }
            }
        }
    }
    if ((a.dft_mask >> lev) & 1u) {
        // the fields of NTFF face cells go to the staging area (dft_flush_2d
        // sums them); a cell lies on at most one x face and one y face
        if (row.face) {
            const int yface = r == a.nt_lo[1] ? 2 : (r == a.nt_hi[1] ? 3 : -1);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int x = cx.x + c;
                if (x < a.nt_lo[0] || x > a.nt_hi[0]) continue;
                float *st = a.stage[lev];
                const float v0 = c ? un(F[0]).y : un(F[0]).x, v1 = c ? un(F[1]).y : un(F[1]).x,
                            v2 = c ? un(F[2]).y : un(F[2]).x;
                if (yface > 0) stage3(st + a.xs_start[yface] + (x - a.nt_lo[0]), a.xs_n, v0, v1, v2);
                const int xface = x == a.nt_lo[0] ? 0 : (x == a.nt_hi[0] ? 1 : -1);
                if (xface >= 0) stage3(st + a.xs_start[xface] + (r - a.nt_lo[1]), a.xs_n, v0, v1, v2);
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) T[s] = third2(F[s]);
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const bool e = s < NE;
            P2 eq;
            if (i == 0) {
                if (e || MU) {
                    const P2 d = sub2(m[s], F[s]);
                    eq = add2(d, d);
                } else {
                    eq = both(0.f);
                }
            } else {
                const int c = slot_comp<MODE>(s), b = cross_slot<MODE>(i, c, e);
                if (b < 0) eq = T[s];
                else if ((cross_sign(i, c) > 0) == e) eq = sub2(T[s], T[b]);
                else eq = add2(T[s], T[b]);
            }
            f[3 * i + s] = sub2(eq, f[3 * i + s]);
        }
    // the absorbing layer and the incident source of dielectric cells, where
    // some cell of the warp's row has one: f* = (f* + source) keep with a zero
    // source and keep = 1 elsewhere
    if (!row.special) return;
    const int dy = min(r, a.ny - 1 - r);
    const float2 ie = un(ie2), im = un(im2);
    const bool diel = a.tfsf && (ie.x != 1.f || ie.y != 1.f || (MU && (im.x != 1.f || im.y != 1.f)));
    const P2 keep = pk(layer_keep(min(cx.dx0, dy), a.w, a.sigma_max, a.inv_w),
                       layer_keep(min(cx.dx1, dy), a.w, a.sigma_max, a.inv_w));
    const bool row_in = r >= a.tf_lo[1] && r <= a.tf_hi[1];
    const bool s0 = diel && row_in && (ie.x != 1.f || (MU && im.x != 1.f)) && cx.x >= a.tf_lo[0] && cx.x <= a.tf_hi[0];
    const bool s1 =
        diel && row_in && (ie.y != 1.f || (MU && im.y != 1.f)) && cx.x + 1 >= a.tf_lo[0] && cx.x + 1 <= a.tf_hi[0];
    if (__any_sync(kAll, s0 || s1)) {
        P2 d[3], d3[3];
        const int l0 = a.inc_axis == 0 ? cx.x : r, l1 = a.inc_axis == 0 ? cx.x + 1 : r;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const bool e = s < NE;
            d[s] = d3[s] = both(0.f);
            if (!e && !MU) continue;
            const float *lm = a.lm[lev] + (size_t)s * a.n_line;
            float v0 = 0.f, v1 = 0.f;
            if (s0) v0 = lm[l0] * (((e ? ie.x : im.x) - 1.0f) * a.inv_scale);
            if (s1) v1 = lm[l1] * (((e ? ie.y : im.y) - 1.0f) * a.inv_scale);
            d[s] = pk(v0, v1);
            d3[s] = third2(d[s]);
        }
#pragma unroll
        for (int i = 0; i < 7; ++i)
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const bool e = s < NE;
                P2 src;
                if (i == 0) {
                    if (!e && !MU) continue;
                    src = mul2(d[s], both(-2.f));
                } else {
                    const int c = slot_comp<MODE>(s), b = cross_slot<MODE>(i, c, e);
                    // e: dE/3 - c x dH/3 (dH only with a mu_r map); h: dH/3 + c x dE/3
                    const bool cross = b >= 0 && (e ? MU : true), own = e || MU;
                    if (!cross && !own) continue;
                    if (!cross) src = d3[s];
                    else if ((cross_sign(i, c) > 0) == e) src = own ? sub2(d3[s], d3[b]) : sub2(both(0.f), d3[b]);
                    else src = own ? add2(d3[s], d3[b]) : d3[b];
                }
                f[3 * i + s] = add2(f[3 * i + s], src);
            }
    }
#pragma unroll
    for (int q = 0; q < 21; ++q) f[q] = mul2(f[q], keep);
}

// Level n of the row a warp takes next waits in shared memory: per lane its two
// cells' pair groups, singles, 1/eps_r (and 1/mu_r), copied by cp.async while
// the warp is at the row before and read by the lane that copied them.  The +y
// group comes from the row above, the -y group from the row below (clamped, Eq. 4).
template <class S, bool MU> struct Stage {
    static constexpr int PB = 4 * (int)sizeof(S), SB = 2 * (int)sizeof(S);  // bytes of two cells' pairs / singles
    static constexpr int S_OFF = 7 * 32 * PB, E_OFF = S_OFF + 7 * 32 * SB, M_OFF = E_OFF + 32 * 8;
    static constexpr int BYTES = M_OFF + (MU ? 32 * 8 : 0);
};
template <class S, bool MU> constexpr int march_smem() { return YBuf<S>::BYTES + kRows * Stage<S, MU>::BYTES; }

template <class S, bool MU>
__device__ __forceinline__ void stage_row(const MarchArgs &a, uint32_t at, int lane, int r, int xc)
{
    using G = Stage<S, MU>;
    const int c = r * a.nxp + xc;
    const int up = r > 0 ? c - a.nxp : c, dn = r < a.ny - 1 ? c + a.nxp : c;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const int k = i == 3 ? up : (i == 4 ? dn : c);
        copy_async<G::PB>(at + (i * 32 + lane) * G::PB, static_cast<const S *>(a.fin[2 * i]) + 2LL * k);
        copy_async<G::SB>(at + G::S_OFF + (i * 32 + lane) * G::SB, static_cast<const S *>(a.fin[2 * i + 1]) + k);
    }
    copy_async<8>(at + G::E_OFF + lane * 8, a.inv_eps + c);
    if constexpr (MU) copy_async<8>(at + G::M_OFF + lane * 8, a.inv_mu + c);
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <class S, bool MU>
__device__ __forceinline__ void take_row(const unsigned char *st, int lane, Dir2<S> d[7], P2 &ie, P2 &im)
{
    using G = Stage<S, MU>;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        if constexpr (sizeof(S) == 4) {
            const float4 v = reinterpret_cast<const float4 *>(st)[i * 32 + lane];
            d[i].c[0] = pk(v.x, v.z);
            d[i].c[1] = pk(v.y, v.w);
            d[i].c[2] = reinterpret_cast<const P2 *>(st + G::S_OFF)[i * 32 + lane];
        } else {
            const uint2 v = reinterpret_cast<const uint2 *>(st)[i * 32 + lane];
            d[i].c[0] = __byte_perm(v.x, v.y, 0x5410);
            d[i].c[1] = __byte_perm(v.x, v.y, 0x7632);
            d[i].c[2] = reinterpret_cast<const unsigned *>(st + G::S_OFF)[i * 32 + lane];
        }
    }
    ie = reinterpret_cast<const P2 *>(st + G::E_OFF)[lane];
    if constexpr (MU) im = reinterpret_cast<const P2 *>(st + G::M_OFF)[lane];
}

// ---- the incident line, several steps in a warp's registers
// A lane holds one node; nodes at the warp's ends go stale one per step, so a
// warp advances 32 - 2 steps nodes.  Writes the node's populations at the
// times that are kept and, for every time, its moments (E, then H components),
// which are all that the lattice reads.
template <int MODE>
__device__ __noinline__ void line_march(const LineMarch &l, int warp)
{
    using PL = Planes<MODE>;
    constexpr int Q = PL::Q, NC = PL::NC;
    const int lane = threadIdx.x & 31, n = l.n;
    const int s = warp * (32 - 2 * l.steps) - l.steps + lane;
    const bool own = lane >= l.steps && lane < 32 - l.steps && s < n;
    const int sc = min(max(s, 0), n - 1);
    if (l.dft_mask && own) {
        // DFT of the line's fields at the times the lattice's pass computes
        for (int c = 0; c < PL::NE; ++c) {
            const int comp = Mode<MODE>::ec(c);
            double re = l.dft[(s * 3 + comp) * 2], im = l.dft[(s * 3 + comp) * 2 + 1];
            for (int k = 0; k < K; ++k) {
                if (!((l.dft_mask >> k) & 1u)) continue;
                const double v = l.dft_scale * (double)l.lm_now[k][(size_t)c * n + s];
                re = fma(v, l.dft_c[k], re);
                im = fma(-v, l.dft_s[k], im);
            }
            l.dft[(s * 3 + comp) * 2] = re;
            l.dft[(s * 3 + comp) * 2 + 1] = im;
        }
    }
    float f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q] = l.from[(size_t)q * n + sc];
    auto moments_out = [&](float *out) {
        if (!out || !own) return;
        float v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = 0.f;
#pragma unroll
        for (int q = 0; q < Q; ++q) v[plane_slot(MODE, q)] += f[q];
#pragma unroll
        for (int c = 0; c < NC; ++c) out[(size_t)c * n + s] = v[c];
    };
    moments_out(l.lm_from);
    const float keep = layer_keep(min(s, n - 1 - s), l.w, l.sigma_max, l.inv_w);
    for (int k = 0; k < l.steps; ++k) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int i = PL::dir(q);
            if (dir_axis(i) < 0 || dir_axis(i) > 1) continue;
            if (dir_axis(i) != l.axis) continue;
            const float v = dir_sign(i) > 0 ? __shfl_up_sync(kAll, f[q], 1) : __shfl_down_sync(kAll, f[q], 1);
            if (s != (dir_sign(i) > 0 ? 0 : n - 1)) f[q] = v;
        }
        float D[3], E[3], H[3];
        moments<MODE>(f, 1.f, D, E, H);
        collide<MODE>(f, D, E, H);
#pragma unroll
        for (int q = 0; q < Q; ++q) f[q] *= keep;
        if (s == l.src_index) {
            // vacuum equilibrium of the prescribed incident fields
            constexpr float sixth = 1.0f / 6.0f;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i = PL::dir(q), c = PL::comp(q);
                if (i == 0) f[q] = 0.f;
                else if (PL::fam(q) == 0) f[q] = (l.src_E[k][c] - cross_c(i, l.src_H[k], c)) * sixth;
                else f[q] = (l.src_H[k][c] + cross_c(i, l.src_E[k], c)) * sixth;
            }
        }
        moments_out(l.lm[k]);
        if (l.full[k] && own)
#pragma unroll
            for (int q = 0; q < Q; ++q) l.full[k][(size_t)q * n + s] = f[q];
    }
}

template <int MODE> __global__ void __launch_bounds__(32) line_start_kernel(const __grid_constant__ LineMarch l)
{
    line_march<MODE>(l, blockIdx.x);
}

// A pass of N steps.
template <int MODE, class S, bool MU, bool REC, int N>
__global__ void __launch_bounds__(32 * kRows, 16 / kRows) march_kernel(const __grid_constant__ MarchArgs a)
{
    using Y = YBuf<S>;
    extern __shared__ __align__(16) unsigned char ybuf[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    chain_release();
    if ((int)blockIdx.x < a.line_blocks) {
        chain_wait();
        const int k = blockIdx.x * kRows + w;
        if (k < a.line_warps) line_march<MODE>(a.line, k);
        return;
    }
    const int bid = blockIdx.x - a.line_blocks;
    const int strip = bid % a.strips, chunk = bid / a.strips;
    const Cols cx = make_cols(strip, lane, a.nx, a.nt_lo, a.nt_hi);
    const Ends ends = make_ends(strip, cx, a.nx);
    const int xc = min(max(cx.x, 0), a.nxp - 2);  // loads stay inside the row
    // owned rows [y0, y1); level n+1 runs over [pa, pend]
    const int y0 = chunk * a.rows, y1 = min(a.ny, y0 + a.rows);
    const int pa = max(y0 - (N - 1), 0), pend = min(y1 - 1 + (N - 1), a.ny - 1);
    __shared__ __align__(8) unsigned long long done[kRows][K];
    init_rows(done);
    chain_wait();

    Dir2<S> d[7];               // this warp's row, in storage form between levels
    P2 ie = both(1.f), im = both(1.f);
    int r = pa + w;             // its row
    unsigned char *stage = ybuf + Y::BYTES + w * Stage<S, MU>::BYTES;
    if (r <= pend) stage_row<S, MU>(a, smem_u32(stage), lane, r, xc);
    if (r > pend) block_sync();  // a warp without a row
    const int above = w == 0 ? kRows - 1 : w - 1, below = w == kRows - 1 ? 0 : w + 1;
    while (r <= pend) {
        take_row<S, MU>(stage, lane, d, ie, im);
        if (r + kRows <= pend) stage_row<S, MU>(a, smem_u32(stage), lane, r + kRows, xc);
        RowFacts row;
        row.r = r;
        row.mine = cx.own && r >= y0 && r < y1;
        row.face = row.mine && r >= a.nt_lo[1] && r <= a.nt_hi[1] &&
                   (cx.xface || r == a.nt_lo[1] || r == a.nt_hi[1]);
        {
            const float2 e = un(ie), m = un(im);
            const bool diel = a.tfsf && (e.x != 1.f || e.y != 1.f || (MU && (m.x != 1.f || m.y != 1.f)));
            row.special = __any_sync(kAll, diel || min(cx.dmin, min(r, a.ny - 1 - r)) < a.w);
        }
#pragma unroll 1
        for (int l = 0; l < N; ++l) {
            if (l > 0 && !await_rows(done, w, l, r - pa, r == pend, N)) {
                give_up(a.status, lane);
                return;
            }
            if (r >= y0 - (N - 1 - l) && r <= y1 - 1 + (N - 1 - l)) {
                from_left<S>(d[1], ends);
                from_right<S>(d[2], ends);
                if (l > 0) {
                    // Eq. 4: the first and last row pull their own groups
                    if (r > 0) d[3] = Y::get(Y::at(ybuf, above, l - 1, 0), lane);
                    if (r < a.ny - 1) d[4] = Y::get(Y::at(ybuf, below, l - 1, 1), lane);
                }
                P2 f[21];
#pragma unroll
                for (int i = 0; i < 7; ++i) from_dir<S>(d[i], f + 3 * i);
                update2<MODE, MU, REC>(a, f, l, cx, row, ie, im);
#pragma unroll
                for (int i = 0; i < 7; ++i) d[i] = to_dir<S>(f + 3 * i);
                if (N == 2 && l == 0 && !await_slot(done, w, r - pa)) {
                    give_up(a.status, lane);
                    return;
                }
                if (l < N - 1) {
                    Y::put(Y::at(ybuf, w, l, 0), lane, d[3]);
                    Y::put(Y::at(ybuf, w, l, 1), lane, d[4]);
                } else if (cx.own) {
                    store_row<S>(a.fout, r * a.nxp + cx.x, cx.x + 1 < a.nx, d);
                }
            }
            publish(&done[w][l]);
        }
        r += kRows;
    }
}

// Sums the staged face fields of cnt steps into the FP64 DFT accumulators in
// step order, one thread per face cell and component, with the fma of the
// single step's direct update.
__global__ void __launch_bounds__(128) dft_flush_2d_kernel(const __grid_constant__ DftFlush2dArgs a)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 3 * a.n) return;
    const int s = (int)(e / a.n);
    const long long j = e - s * a.n;
    int f = 0;
    while (f + 1 < 4 && j >= a.start[f + 1]) ++f;
    const long long plane = a.plane[f];
    double *base = a.dft + a.face_off[f] + (j - a.start[f]) + 2 * s * plane;
    const float *src = a.stage + e;
    double re = base[0], im = base[plane];
#pragma unroll 8
    for (int k = 0; k < a.cnt; ++k) {
        const double v = (double)src[(long long)k * 3 * a.n];
        re = fma(v, a.sc[k], re);
        im = fma(v, -a.ss[k], im);
    }
    base[0] = re;
    base[plane] = im;
}

// ---- host side
std::mutex g_march_mu;
int g_march_bps[kMaxDevices][2][3][2][2][K + 1];
template <class S> constexpr int storage_slot() { return std::is_same<S, float>::value ? 0 : (std::is_same<S, __half>::value ? 1 : 2); }

template <int MODE, class S, bool MU, bool REC, int N>
cudaError_t launch_march_t(MarchArgs a, int share, cudaStream_t s)
{
    int dev = 0, bps = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(g_march_mu);
        int &got = g_march_bps[dev][MODE][storage_slot<S>()][MU][REC][N];
        e = march_setup_kernel(march_kernel<MODE, S, MU, REC, N>, march_smem<S, MU>(), got);
        if (e != cudaSuccess) return e;
        bps = got;
    }
    a.strips = (a.nx + kStrip - 1) / kStrip;
    a.rows = march_rows(a.ny, a.strips, std::max<long long>(1, (long long)std::max(1, sm_count()) * bps / share), N == 2);
    const long long chunks = (a.ny + a.rows - 1) / a.rows;
    a.line_warps = a.line.steps > 0 ? line_march_warps(a.line) : 0;
    a.line_blocks = (a.line_warps + kRows - 1) / kRows;
    const long long blocks = a.line_blocks + chunks * a.strips;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    return launch_chained(a.chain != 0 && share == 1, march_kernel<MODE, S, MU, REC, N>, (unsigned)blocks, 32 * kRows, march_smem<S, MU>(), s, a);
}

template <int MODE, class S, bool MU>
cudaError_t launch_march_steps(bool rec, const MarchArgs &a, int share, cudaStream_t s)
{
    static_assert(K == 4, "one case each");
    if constexpr (std::is_same<S, float>::value && !MU) {
        if (rec && a.steps == K) return launch_march_t<MODE, S, MU, true, K>(a, share, s);
    }
    if (rec) return cudaErrorInvalidValue;
    switch (a.steps) {
    case 2: return launch_march_t<MODE, S, MU, false, 2>(a, share, s);
    case 3: return launch_march_t<MODE, S, MU, false, 3>(a, share, s);
    case K: return launch_march_t<MODE, S, MU, false, K>(a, share, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int MODE>
cudaError_t launch_march_mode(int storage, bool mu, bool rec, const MarchArgs &a, int share, cudaStream_t s)
{
    switch (storage * 2 + (mu ? 1 : 0)) {
    case 0: return launch_march_steps<MODE, float, false>(rec, a, share, s);
    case 1: return launch_march_steps<MODE, float, true>(rec, a, share, s);
    case 2: return launch_march_steps<MODE, __half, false>(rec, a, share, s);
    case 3: return launch_march_steps<MODE, __half, true>(rec, a, share, s);
    case 4: return launch_march_steps<MODE, __nv_bfloat16, false>(rec, a, share, s);
    case 5: return launch_march_steps<MODE, __nv_bfloat16, true>(rec, a, share, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int line_march_warps(const LineMarch &l) { return (l.n + 31 - 2 * l.steps) / (32 - 2 * l.steps); }

bool march_fits(int mode, int nx, int ny, int nz) { return mode != 2 && nz == 1 && nx >= 2 && ny >= 2; }

cudaError_t launch_march(int mode, int storage, const MarchArgs &a, bool rec, int share, cudaStream_t s)
{
    if (a.nxp % 32 || !march_fits(mode, a.nx, a.ny, 1)) return cudaErrorInvalidValue;
    share = std::max(1, share);
    return mode == 0 ? launch_march_mode<0>(storage, a.inv_mu != nullptr, rec, a, share, s)
                     : launch_march_mode<1>(storage, a.inv_mu != nullptr, rec, a, share, s);
}

cudaError_t launch_line_start(int mode, const LineMarch &l, cudaStream_t s)
{
    const int warps = line_march_warps(l);
    if (mode == 0) line_start_kernel<0><<<warps, 32, 0, s>>>(l);
    else line_start_kernel<1><<<warps, 32, 0, s>>>(l);
    return cudaGetLastError();
}

cudaError_t launch_dft_flush_2d(const DftFlush2dArgs &a, cudaStream_t s)
{
    if (a.cnt < 1 || a.cnt > kMarchStage || a.n <= 0) return cudaErrorInvalidValue;
    dft_flush_2d_kernel<<<(unsigned)((3 * a.n + 127) / 128), 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace lbem
