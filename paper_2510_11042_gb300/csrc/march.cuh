// Device code shared by the 2D passes of four steps: the forward pass (march.cu)
// and its transpose (march_adjoint.cu).  Internal to liblbem (internal linkage
// in each translation unit that includes it).
#pragma once

#include "step_cell.cuh"

namespace lbem {
namespace {

constexpr int K = kMarchSteps;
constexpr int kStrip = 64 - 2 * K;   // owned cells of a warp along x
constexpr int kEdgeLanes = K / 2;    // lanes on each side that own no cell
constexpr int kRows = 16;            // warps of a block, rows in flight
static_assert(K % 2 == 0, "a lane's two cells are both owned or both not");

// ---- packed FP32 arithmetic over a lane's two cells.  A pair lives in one
// 64-bit register throughout: as a float2 its halves were moved in and out of
// register pairs around every packed instruction (105 moves a row and level).
using P2 = unsigned long long;
__device__ __forceinline__ P2 pk(float x, float y)
{
    P2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 un(P2 v)
{
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}
__device__ __forceinline__ P2 both(float v) { return pk(v, v); }
__device__ __forceinline__ P2 add2(P2 a, P2 b)
{
    P2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b)
{
    P2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c)
{
    P2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// a - b, rounded once (the product with -1 is exact)
__device__ __forceinline__ P2 sub2(P2 a, P2 b) { return fma2(b, both(-1.f), a); }
__device__ __forceinline__ P2 third2(P2 x) { return fma2(x, both(kThirdHi), mul2(x, both(kThirdLo))); }

// ---- one direction's three values of a lane's two cells in storage form: each
// slot of both cells (16-bit: as a packed pair)
template <class S> struct Dir2 { unsigned c[3]; };
template <> struct Dir2<float> { P2 c[3]; };

template <class S> __device__ __forceinline__ Dir2<S> to_dir(const P2 *f)
{
    Dir2<S> d;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if constexpr (sizeof(S) == 4) {
            d.c[k] = f[k];
        } else {
            const float2 v = un(f[k]);
            d.c[k] = Io<S>::pack(v.x, v.y);
        }
    }
    return d;
}

template <class S> __device__ __forceinline__ void from_dir(const Dir2<S> &d, P2 *f)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if constexpr (sizeof(S) == 4) {
            f[k] = d.c[k];
        } else {
            const float2 v = Io<S>::unpack(d.c[k]);
            f[k] = pk(v.x, v.y);
        }
    }
}

constexpr unsigned kAll = 0xffffffffu;

// Where a warp's cells meet the grid's x ends: whether any do (uniform over
// the warp), and this lane's first cell at x == 0, its first or second at nx - 1.
struct Ends { bool any, first0, last0, last1; };

// The pull of the +x group: each cell's value from the cell to its left; at
// x == 0 the cell's own (Eq. 4).
template <class S> __device__ __forceinline__ void from_left(Dir2<S> &d, const Ends &e)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if constexpr (sizeof(S) == 4) {
            const float2 v = un(d.c[k]);
            float l = __shfl_up_sync(kAll, v.y, 1);
            if (e.any) {
                asm volatile("");  // a branch, not selects in every strip
                if (e.first0) l = v.x;
            }
            d.c[k] = pk(l, v.x);
        } else {
            unsigned l = __shfl_up_sync(kAll, d.c[k], 1) >> 16;
            if (e.any && e.first0) l = d.c[k];
            d.c[k] = __byte_perm(l, d.c[k], 0x5410);
        }
    }
}

// The pull of the -x group: from the cell to the right; at x == nx - 1 the
// cell's own.
template <class S> __device__ __forceinline__ void from_right(Dir2<S> &d, const Ends &e)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if constexpr (sizeof(S) == 4) {
            const float2 v = un(d.c[k]);
            float r = __shfl_down_sync(kAll, v.x, 1), m = v.y;
            if (e.any) {
                asm volatile("");
                if (e.last0) m = v.x;
                if (e.last1) r = v.y;
            }
            d.c[k] = pk(m, r);
        } else {
            unsigned r = __shfl_down_sync(kAll, d.c[k], 1), m = d.c[k] >> 16;
            if (e.any) {
                if (e.last0) m = d.c[k];
                if (e.last1) r = d.c[k] >> 16;
            }
            d.c[k] = __byte_perm(m, r, 0x5410);
        }
    }
}

// ---- +-y groups of the rows in flight, in shared memory: row slot w holds the
// +y and -y groups of levels n+1 .. n+K-1 of the row its warp is at.
template <class S> struct YBuf {
    static constexpr int V = sizeof(S) == 4 ? 16 : 8;       // bytes of slots 0, 1 of a lane's two cells
    static constexpr int GROUP = 32 * (V + V / 2);
    static constexpr int BYTES = kRows * 2 * (K - 1) * GROUP;
    // up = 0: the +y group, 1: the -y group
    __device__ static unsigned char *at(unsigned char *sm, int w, int lev, int up)
    {
        return sm + ((w * (K - 1) + lev) * 2 + up) * GROUP;
    }
    __device__ static void put(unsigned char *g, int lane, const Dir2<S> &d)
    {
        if constexpr (sizeof(S) == 4) {
            reinterpret_cast<ulonglong2 *>(g)[lane] = make_ulonglong2(d.c[0], d.c[1]);
            reinterpret_cast<P2 *>(g + 32 * V)[lane] = d.c[2];
        } else {
            reinterpret_cast<uint2 *>(g)[lane] = make_uint2(d.c[0], d.c[1]);
            reinterpret_cast<unsigned *>(g + 32 * V)[lane] = d.c[2];
        }
    }
    __device__ static Dir2<S> get(const unsigned char *g, int lane)
    {
        Dir2<S> d;
        if constexpr (sizeof(S) == 4) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(g)[lane];
            d.c[0] = v.x;
            d.c[1] = v.y;
            d.c[2] = reinterpret_cast<const P2 *>(g + 32 * V)[lane];
        } else {
            const uint2 v = reinterpret_cast<const uint2 *>(g)[lane];
            d.c[0] = v.x;
            d.c[1] = v.y;
            d.c[2] = reinterpret_cast<const unsigned *>(g + 32 * V)[lane];
        }
        return d;
    }
};

// The block barrier that every warp passes once, at places of its own.
__device__ __forceinline__ void block_sync() { asm volatile("barrier.cta.sync 1;" ::: "memory"); }

// One mbarrier per row slot and level: its phase m completes when the slot's
// m-th row has done the level.  A wait is bounded: kPolls polls of up to
// kSuspendNs each, for which the hardware suspends the warp.
constexpr int kPolls = 1 << 18;
constexpr unsigned kSuspendNs = 4000;
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void publish(const unsigned long long *bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool reached(uint32_t bar, uint32_t phase)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(phase & 1), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool await(const unsigned long long *bar, uint32_t phase)
{
    const uint32_t at = smem_u32(bar);
    for (int k = 0; k < kPolls; ++k)
        if (reached(at, phase)) return true;
    return false;
}

// Component of slot s, and the slot of a component (-1: not carried).
template <int MODE> __device__ __forceinline__ constexpr int slot_comp(int s)
{
    return s < Planes<MODE>::NE ? Mode<MODE>::ec(s) : Mode<MODE>::hc(s - Planes<MODE>::NE);
}
// cross_c(i, V, a) as sign times V[b]: sign 0 where it vanishes or the mode does not carry V[b]
template <int MODE> __device__ __forceinline__ constexpr int cross_slot(int i, int a, bool of_h)
{
    const int d = dir_axis(i);
    if (a == d) return -1;
    return of_h ? slot_H(MODE, 3 - a - d) : slot_E(MODE, 3 - a - d);
}
__device__ __forceinline__ constexpr int cross_sign(int i, int a)
{
    return dir_sign(i) * (a == (dir_axis(i) + 2) % 3 ? 1 : -1);
}

// What a lane knows of its two columns.
struct Cols {
    int x;          // of the first cell (even; may lie outside the grid)
    int dx0, dx1;   // distance to the nearer x face
    int dmin;       // the smaller of them
    bool own;       // the strip owns the cells
    bool xface;     // one of them lies on an x face of the NTFF box
};

// What a warp knows of its row, the same at all its levels.
struct RowFacts {
    int r;
    bool mine;      // the lane's cells are owned by this strip and chunk
    bool special;   // some cell of the warp's needs more than the plain update (uniform)
    bool face;      // a cell of the lane lies on the NTFF box
};

__device__ __forceinline__ Cols make_cols(int strip, int lane, int nx, const int nt_lo[2], const int nt_hi[2])
{
    Cols c;
    c.x = strip * kStrip - K + 2 * lane;
    c.dx0 = min(c.x, nx - 1 - c.x);
    c.dx1 = min(c.x + 1, nx - 2 - c.x);
    c.dmin = min(c.dx0, c.dx1);
    c.own = lane >= kEdgeLanes && lane < 32 - kEdgeLanes && c.x < nx;
    c.xface = c.x == nt_lo[0] || c.x == nt_hi[0] || c.x + 1 == nt_lo[0] || c.x + 1 == nt_hi[0];
    return c;
}
__device__ __forceinline__ Ends make_ends(int strip, const Cols &c, int nx)
{
    Ends e;
    e.any = strip == 0 || strip * kStrip - K + 63 >= nx - 1;
    e.first0 = c.x == 0;
    e.last0 = c.x == nx - 1;
    e.last1 = c.x + 1 == nx - 1;
    return e;
}

// The waits of level l > 0 of row r (index i of the chunk's, the last one with
// last set) in a pass of n levels: level l - 1 of the rows above and below.  The
// same waits (also where the level itself is not computed, in the chunk's first
// and last rows) keep the groups of row r until both neighbours have read them:
// row r + kRows, which takes their place, starts once row r is finished, so both
// have read its groups but those of level n - 2; and it reaches that level once
// the rows beside it are under way, whose warps have then finished the rows beside
// r.  (With two levels it is the first one, which has no waits of its own:
// await_slot.)  The last row, which has none below it, waits for the row kRows - 1
// before it in that one's stead.
// A wait tells a phase only from its neighbours, so no warp may wait for a
// slot's second row before the slot's first has begun: the block barrier.
__device__ __forceinline__ bool await_rows(unsigned long long (*done)[K], int w, int l, int i, bool last, int n)
{
    const int above = w == 0 ? kRows - 1 : w - 1, below = w == kRows - 1 ? 0 : w + 1;
    if (l == 1 && i < kRows) block_sync();
    bool ok = i == 0 || await(&done[above][l - 1], (uint32_t)(i - 1) / kRows);
    if (!last) ok = ok && await(&done[below][l - 1], (uint32_t)(i + 1) / kRows);
    else if (i >= kRows - 1) ok = ok && await(&done[below][n - 1], (uint32_t)(i - (kRows - 1)) / kRows);
    return __all_sync(kAll, ok);
}
// The wait of a row's first level in a pass of two, before its groups are
// written: the rows beside the one whose place they take (i - kRows) are finished.
__device__ __forceinline__ bool await_slot(unsigned long long (*done)[K], int w, int i)
{
    if (i < kRows) return true;
    const int above = w == 0 ? kRows - 1 : w - 1, below = w == kRows - 1 ? 0 : w + 1;
    const bool ok = (i == kRows || await(&done[above][1], (uint32_t)(i - kRows - 1) / kRows)) &&
                    await(&done[below][1], (uint32_t)(i - kRows + 1) / kRows);
    return __all_sync(kAll, ok);
}
__device__ __forceinline__ void init_rows(unsigned long long (*done)[K])
{
    if (threadIdx.x < kRows * K)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done[0][0] + threadIdx.x)) : "memory");
    __syncthreads();
}


template <int N> __device__ __forceinline__ void copy_async(uint32_t dst, const void *src)
{
    if constexpr (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(N) : "memory");
}

// A warp whose wait ran out: the error flag, then the end of its own copies.
__device__ __forceinline__ void give_up(int *status, int lane)
{
    if (lane == 0) atomicOr(status, 1);
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <class S>
__device__ __forceinline__ void store_row(void *const *fout, int c, bool two, const Dir2<S> d[7])
{
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        void *p = fout[2 * i], *q = fout[2 * i + 1];
        if constexpr (sizeof(S) == 4) {
            const float2 u = un(d[i].c[0]), v = un(d[i].c[1]);
            if (two) {
                *reinterpret_cast<float4 *>(static_cast<float2 *>(p) + c) = make_float4(u.x, v.x, u.y, v.y);
                *reinterpret_cast<P2 *>(static_cast<float *>(q) + c) = d[i].c[2];
            } else {
                static_cast<float2 *>(p)[c] = make_float2(u.x, v.x);
                static_cast<float *>(q)[c] = un(d[i].c[2]).x;
            }
        } else {
            const unsigned u = __byte_perm(d[i].c[0], d[i].c[1], 0x5410), v = __byte_perm(d[i].c[0], d[i].c[1], 0x7632);
            if (two) {
                *reinterpret_cast<uint2 *>(static_cast<unsigned *>(p) + c) = make_uint2(u, v);
                *reinterpret_cast<unsigned *>(static_cast<unsigned short *>(q) + c) = d[i].c[2];
            } else {
                static_cast<unsigned *>(p)[c] = u;
                static_cast<unsigned short *>(q)[c] = (unsigned short)(d[i].c[2] & 0xffffu);
            }
        }
    }
}

// Rows per chunk of a grid ny rows high and strips wide, cap resident blocks:
// whole waves; a chunk of L rows takes about L + 12 rows' time (its recomputed
// rows and the start of its pipeline).  The last wave waits for its slowest chunk
// (the scatterer's, whose cells take the incident source, or one that falls behind
// on a long march), which counts as kSlowest of a wave more: one wave of long
// chunks is worse than several of shorter ones.  us a step, one wave -> as chosen:
// 4096^2 EZ FP16 176 -> 143, FP32 147 -> 132, 2800^2 FP32 85.5 -> 63.9, 1300^2 FP32
// 20.7 -> 18.3; the batched sweep of 32 cylinders (a quarter of the blocks each)
// 19.3 -> 17.1 ms.  The count that is best without it stays where it costs less than
// 3 % more: there several waves measured between 10 % slower (1024^2: 12.2 in one
// wave, 13.5 in two) and no better (3400^2: 90.6 in five, 92.5 in seven).
// Passes of two levels, which have the least work to a byte, like shorter chunks
// still (4096^2 EZ with kSlowest -> kSlowestTwo: FP16 186 -> 178, FP32 240 -> 226).
constexpr double kSlowest = 0.18, kSlowestTwo = 0.6, kStay = 1.03;
inline int march_rows(int ny, int strips, long long cap, bool two = false)
{
    const double slowest = two ? kSlowestTwo : kSlowest;
    struct Plan { long long chunks; double waves, rows; } plain = {0, 0, 0}, best = {0, 0, 0};
    auto cost = [](const Plan &p, double extra) { return (p.waves + extra) * (p.rows + 12.0); };
    for (long long w = 1; w <= 256; ++w) {
        const long long c = std::max<long long>(1, w * cap / strips);
        const long long rows = std::max<long long>(kMarchMinRows, (ny + c - 1) / c);
        const long long n = (ny + rows - 1) / rows;
        const Plan p = {n, (double)((n * strips + cap - 1) / cap), (double)rows};
        if (plain.chunks == 0 || cost(p, 0.0) < cost(plain, 0.0)) plain = p;
        if (best.chunks == 0 || cost(p, slowest) < cost(best, slowest)) best = p;
        if (rows <= kMarchMinRows) break;
    }
    const long long chunks = (cost(plain, slowest) < kStay * cost(best, slowest) ? plain : best).chunks;
    return (int)std::max<long long>((ny + chunks - 1) / chunks, kMarchMinRows);
}

// A pass kernel's shared-memory opt-in and resident blocks per SM, once per
// device (bps: the caller's cache entry for the current device).
template <class Kernel> cudaError_t march_setup_kernel(Kernel k, int smem, int &bps)
{
    if (bps > 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32 * kRows, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaErrorInvalidConfiguration;
    bps = n;
    return cudaSuccess;
}

}  // namespace
}  // namespace lbem
