// Four steps of the discrete adjoint per pass in 2D (FP32): the transpose of
// the forward pass of march.cu, in the same form -- a block marches along y, a
// warp carries a row through the four levels in registers, two cells to a lane
// (march.cuh).  One level is adjoint_step_kernel's update (adjoint.cu):
//     m = K lambda, lambda = S^T mu   (transposed clamped pull, as a gather)
//     A = sum_i (m_ei - c_i x m_hi)/3 - 2 m_e0 + dJ/dE|DFT,  Bv likewise
//     mu_e = beta A + 2 m_e0 - m_e,  mu_h = Bv - m_h,  dJ/dbeta += A . D
// A direction's group comes from the cell its velocity points to, so +x comes
// from the right, +y from the row below, and the cells that the clamp maps
// back onto themselves add their own.  A row's gradient stays in FP64 registers
// over the four levels; the recorded D of the four steps is copied with the row.
//
// Bound as the forward pass on small grids: instruction issue and the rows'
// waits.  512^2 EZ, us a step: backward, one launch a step 8.3 -> 6.3, and 5.5
// chained to the launch before; replay (march_kernel with the recorded D) 8.3 -> 5.2,
// and 4.6.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "march.cuh"

namespace lbem {
namespace {

// What a warp copies ahead per row: 7 pair groups, 7 singles, 1/eps_r, the
// recorded D of the four steps (NE planes each) and the FP64 gradient.
template <int MODE> struct AdjStage {
    static constexpr int NE = Planes<MODE>::NE;
    static constexpr int S_OFF = 7 * 32 * 16, E_OFF = S_OFF + 7 * 32 * 8, R_OFF = E_OFF + 32 * 8,
                         G_OFF = R_OFF + K * NE * 32 * 8, BYTES = G_OFF + 32 * 16;
    static constexpr int SMEM = YBuf<float>::BYTES + kRows * BYTES;
};

template <int MODE>
__device__ __forceinline__ void stage_row(const MarchAdjointArgs &a, uint32_t at, int lane, int r, int xc)
{
    using G = AdjStage<MODE>;
    const int c = r * a.nxp + xc;
    const int up = r > 0 ? c - a.nxp : c, dn = r < a.ny - 1 ? c + a.nxp : c;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const int k = i == 3 ? dn : (i == 4 ? up : c);  // +y from the row below, -y from the row above
        copy_async<16>(at + (i * 32 + lane) * 16, a.lin[2 * i] + 2LL * k);
        copy_async<8>(at + G::S_OFF + (i * 32 + lane) * 8, a.lin[2 * i + 1] + k);
    }
    copy_async<8>(at + G::E_OFF + lane * 8, a.inv_eps + c);
#pragma unroll
    for (int l = 0; l < K; ++l)
#pragma unroll
        for (int s = 0; s < G::NE; ++s)
            copy_async<8>(at + G::R_OFF + ((l * G::NE + s) * 32 + lane) * 8, a.rec[l] + (long long)s * a.P + c);
    copy_async<16>(at + G::G_OFF + lane * 16, a.grad + c);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// +x group: from the right neighbour (none at nx - 1); at x == 0 also the cell's own.
__device__ __forceinline__ void adj_from_right(Dir2<float> &d, const Ends &e)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 v = un(d.c[k]);
        float m = v.y, r = __shfl_down_sync(kAll, v.x, 1);
        if (e.any) {
            asm volatile("");
            if (e.last0) m = 0.f;
            if (e.last1) r = 0.f;
            if (e.first0) m += v.x;
        }
        d.c[k] = pk(m, r);
    }
}
// -x group: from the left neighbour (none at 0); at nx - 1 also the cell's own.
__device__ __forceinline__ void adj_from_left(Dir2<float> &d, const Ends &e)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 v = un(d.c[k]);
        float l = __shfl_up_sync(kAll, v.y, 1), m = v.x;
        if (e.any) {
            asm volatile("");
            if (e.first0) l = 0.f;
            if (e.last0) l += v.x;
            if (e.last1) m += v.y;
        }
        d.c[k] = pk(l, m);
    }
}

// One adjoint level of a lane's two cells: lambda in, mu out; dg: this step's
// A . D of both cells.
template <int MODE>
__device__ __forceinline__ void adjoint2(const MarchAdjointArgs &a, P2 *f, int lev, const Cols &cx, const RowFacts &row,
                                         P2 beta, const P2 *D, float2 &dg)
{
    constexpr int NE = Planes<MODE>::NE;
    const int r = row.r;
    if (row.special) {
        const int dy = min(r, a.ny - 1 - r);
        const P2 keep = pk(layer_keep(min(cx.dx0, dy), a.w, a.sigma_max, a.inv_w),
                           layer_keep(min(cx.dx1, dy), a.w, a.sigma_max, a.inv_w));
#pragma unroll
        for (int q = 0; q < 21; ++q) f[q] = mul2(f[q], keep);
    }
    P2 A[3];  // by slot: A of the e components, Bv of the h components
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const bool e = s < NE;
        const int c = slot_comp<MODE>(s);
        P2 sum = both(0.f);
#pragma unroll
        for (int i = 1; i < 7; ++i) {
            // e: m_e - c_i x m_h, h: m_h + c_i x m_e
            const int b = cross_slot<MODE>(i, c, e);
            P2 t = f[3 * i + s];
            if (b >= 0) t = ((cross_sign(i, c) > 0) == e) ? sub2(t, f[3 * i + b]) : add2(t, f[3 * i + b]);
            sum = i == 1 ? t : add2(sum, t);
        }
        A[s] = third2(sum);
        if (e) A[s] = fma2(f[s], both(-2.f), A[s]);
    }
    if (((a.dft_mask >> lev) & 1u) && row.face) {
        // dJ/dx(t) = Re(G (cos - j sin)) 2/(P T) for every DFT entry of the cell
        float2 add[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int x = cx.x + c;
            if (x < a.nt_lo[0] || x > a.nt_hi[0]) continue;
            double dx[3] = {0.0, 0.0, 0.0};
            for (int face = 0; face < 4; ++face) {
                if ((face < 2 ? x : r) != (face & 1 ? a.nt_hi[face / 2] : a.nt_lo[face / 2])) continue;
                const long long plane = (long long)a.face_nu[face] * a.face_nv[face];
                const double *base = a.G + a.face_off[face] + (face < 2 ? r - a.nt_lo[1] : x - a.nt_lo[0]);
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    dx[s] += base[(2 * s) * plane] * a.dft_c[lev] + base[(2 * s + 1) * plane] * a.dft_s[lev];
            }
#pragma unroll
            for (int s = 0; s < 3; ++s) (c ? add[s].y : add[s].x) = (float)(a.dft_scale * dx[s]);
        }
#pragma unroll
        for (int s = 0; s < 3; ++s) A[s] = add2(A[s], pk(add[s].x, add[s].y));
    }
    P2 g = both(0.f);
#pragma unroll
    for (int s = 0; s < NE; ++s) g = fma2(A[s], D[s], g);
    dg = un(g);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const P2 v = s < NE ? fma2(beta, A[s], add2(f[s], f[s])) : A[s];
#pragma unroll
        for (int i = 0; i < 7; ++i) f[3 * i + s] = sub2(v, f[3 * i + s]);
    }
}

template <int MODE>
__global__ void __launch_bounds__(32 * kRows, 1) march_adjoint_kernel(const __grid_constant__ MarchAdjointArgs a)
{
    using Y = YBuf<float>;
    using G = AdjStage<MODE>;
    constexpr int NE = G::NE;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(8) unsigned long long done[kRows][K];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int strip = blockIdx.x % a.strips, chunk = blockIdx.x / a.strips;
    const Cols cx = make_cols(strip, lane, a.nx, a.nt_lo, a.nt_hi);
    const Ends ends = make_ends(strip, cx, a.nx);
    const int xc = min(max(cx.x, 0), a.nxp - 2);
    const int y0 = chunk * a.rows, y1 = min(a.ny, y0 + a.rows);
    const int pa = max(y0 - (K - 1), 0), pend = min(y1 - 1 + (K - 1), a.ny - 1);
    chain_release();
    init_rows(done);
    chain_wait();
    unsigned char *stage = smem + Y::BYTES + w * G::BYTES;
    int r = pa + w;
    if (r <= pend) stage_row<MODE>(a, smem_u32(stage), lane, r, xc);
    else block_sync();  // a warp without a row
    const int above = w == 0 ? kRows - 1 : w - 1, below = w == kRows - 1 ? 0 : w + 1;
    while (r <= pend) {
        Dir2<float> d[7];
        P2 D[K][NE];
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const float4 v = reinterpret_cast<const float4 *>(stage)[i * 32 + lane];
            d[i].c[0] = pk(v.x, v.z);
            d[i].c[1] = pk(v.y, v.w);
            d[i].c[2] = reinterpret_cast<const P2 *>(stage + G::S_OFF)[i * 32 + lane];
        }
        const P2 beta = reinterpret_cast<const P2 *>(stage + G::E_OFF)[lane];
#pragma unroll
        for (int k = 0; k < K * NE; ++k) D[k / NE][k % NE] = reinterpret_cast<const P2 *>(stage + G::R_OFF)[k * 32 + lane];
        double2 grad = reinterpret_cast<const double2 *>(stage + G::G_OFF)[lane];
        if (r + kRows <= pend) stage_row<MODE>(a, smem_u32(stage), lane, r + kRows, xc);
        RowFacts row;
        row.r = r;
        row.mine = cx.own && r >= y0 && r < y1;
        row.special = __any_sync(kAll, min(cx.dmin, min(r, a.ny - 1 - r)) < a.w);
        // unlike the forward pass's staging, which one owner does, the source on
        // the NTFF faces enters every copy of a cell
        row.face = r >= a.nt_lo[1] && r <= a.nt_hi[1] && (cx.xface || r == a.nt_lo[1] || r == a.nt_hi[1]);
#pragma unroll 1
        for (int l = 0; l < K; ++l) {
            if (l > 0 && !await_rows(done, w, l, r - pa, r == pend, K)) {
                give_up(a.status, lane);
                return;
            }
            if (r >= y0 - (K - 1 - l) && r <= y1 - 1 + (K - 1 - l)) {
                adj_from_right(d[1], ends);
                adj_from_left(d[2], ends);
                // the row's own +-y groups, which the clamp at the first and last
                // row adds (at l == 0 the copies in d are the neighbours')
                Dir2<float> own;
                const bool edge = r == 0 || r == a.ny - 1;
                if (edge) {
                    const int i = r == 0 ? 3 : 4;
                    if (l > 0) {
                        own = r == 0 ? d[3] : d[4];
                    } else {
                        const long long c = (long long)r * a.nxp + xc;
                        const float4 v = *reinterpret_cast<const float4 *>(a.lin[2 * i] + 2 * c);
                        own.c[0] = pk(v.x, v.z);
                        own.c[1] = pk(v.y, v.w);
                        own.c[2] = *reinterpret_cast<const P2 *>(a.lin[2 * i + 1] + c);
                    }
                }
                if (l > 0) {
                    if (r < a.ny - 1) d[3] = Y::get(Y::at(smem, below, l - 1, 0), lane);
                    if (r > 0) d[4] = Y::get(Y::at(smem, above, l - 1, 1), lane);
                }
                if (edge) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (r == a.ny - 1) d[3].c[k] = both(0.f);
                        if (r == 0) d[4].c[k] = both(0.f);
                        if (r == 0) d[3].c[k] = add2(d[3].c[k], own.c[k]);
                        else d[4].c[k] = add2(d[4].c[k], own.c[k]);
                    }
                }
                P2 f[21], now[NE];
#pragma unroll
                for (int i = 0; i < 7; ++i) from_dir<float>(d[i], f + 3 * i);
#pragma unroll
                for (int s = 0; s < NE; ++s)
                    now[s] = l == 0 ? D[0][s] : (l == 1 ? D[1][s] : (l == 2 ? D[2][s] : D[3][s]));
                float2 dg;
                adjoint2<MODE>(a, f, l, cx, row, beta, now, dg);
                grad.x += (double)dg.x;
                grad.y += (double)dg.y;
#pragma unroll
                for (int i = 0; i < 7; ++i) d[i] = to_dir<float>(f + 3 * i);
                if (l < K - 1) {
                    Y::put(Y::at(smem, w, l, 0), lane, d[3]);
                    Y::put(Y::at(smem, w, l, 1), lane, d[4]);
                } else if (cx.own) {
                    const int c = r * a.nxp + cx.x;
                    const bool two = cx.x + 1 < a.nx;
                    store_row<float>(a.lout, c, two, d);
                    a.grad_out[c] = grad.x;
                    if (two) a.grad_out[c + 1] = grad.y;
                }
            }
            publish(&done[w][l]);
        }
        r += kRows;
    }
}

std::mutex g_adj_mu;
int g_adj_bps[kMaxDevices][2];

template <int MODE> cudaError_t launch_t(MarchAdjointArgs a, cudaStream_t s)
{
    int dev = 0, bps = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(g_adj_mu);
        e = march_setup_kernel(march_adjoint_kernel<MODE>, AdjStage<MODE>::SMEM, g_adj_bps[dev][MODE]);
        if (e != cudaSuccess) return e;
        bps = g_adj_bps[dev][MODE];
    }
    a.strips = (a.nx + kStrip - 1) / kStrip;
    a.rows = march_rows(a.ny, a.strips, (long long)std::max(1, sm_count()) * bps);
    const long long blocks = (long long)((a.ny + a.rows - 1) / a.rows) * a.strips;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    return launch_chained(true, march_adjoint_kernel<MODE>, (unsigned)blocks, 32 * kRows, AdjStage<MODE>::SMEM, s, a);
}

}  // namespace

cudaError_t launch_march_adjoint(int mode, const MarchAdjointArgs &a, cudaStream_t s)
{
    if (a.nxp % 32 || !march_fits(mode, a.nx, a.ny, 1)) return cudaErrorInvalidValue;
    return mode == 0 ? launch_t<0>(a, s) : launch_t<1>(a, s);
}

}  // namespace lbem
