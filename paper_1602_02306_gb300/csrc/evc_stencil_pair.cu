// evc_stencil_pair.cu -- two 7-point stencil passes in one kernel: the factor
//   x <- g^2 ((K - re)^2 + im^2) x     of the Chebyshev preconditioner M = p_d(K)
// in factored form (a conjugate pair of roots; Sec. 6), i.e. the passes
//   u   = insc_c (k1 (L x)_offdiag + (k1 cd + k0) x)
//   out = k1' (L u)_offdiag + (k1' cd + k0') u + a0 xs_c x - ppc_c pp
// with u kept on chip.  FP32; the arithmetic per point is that of the single
// passes in evc_stencil.cu, term by term, so the result is bitwise theirs.
//
// Why: apart, the two passes move five vectors through L2 (x, u, u, x, out) plus
// the arms of 8 x 8 tiles; together two, plus arms twice as wide.
//
// A block owns a TS x TS tile of (x, y) points and 16 of a chunk's 32 columns and
// marches along z.  Tiled tensor copies (cp.async.bulk.tensor) stage, per plane,
// the tile of x with its radius-2 diamond of neighbours in shared memory, every
// arm with its own wrapped coordinate, even and odd x apart so that patches two
// points wide read without bank conflicts.  A thread owns a 2 x 2 patch of points
// and two columns of the tile and a ring of one point around it: it computes u at
// its points (z neighbours in a register window, in-plane neighbours outside the
// patch from the staged plane) and stores them to a plane of u (four in turn);
// from u's window and the neighbours' u of the plane before it computes out.
// Warps arrive at a barrier when their u of a plane is stored and wait for it a
// plane later, so they need not march in step.  The ring's u are computed by every
// tile that needs them: (TS + 2)^2 / TS^2 of the first pass's work.
//
// What bounds it: the shared-memory pipe.  A point costs 6 reads and writes of its
// columns there (own x, 2 x neighbours, u, 2 u neighbours) times the ring, the
// staging and the stores: l1tex 71 % busy, HBM half.  Measured, Chebyshev-8
// operator of one Lanczos step (two M of four pairs, one H pass), us, before
// (best tile shape of the single passes) | now: 64^3, 128 columns 912 | 696; 96^3
// 2894 | 2198; 40^3 256 | 233; 32^3 178 | 147; with the default shapes 64^3 1577 |
// 868, 40^3 498 | 270, 32^3 306 | 195.  Tried: 8 columns per block (32-byte rows:
// the tensor copies become the limit, 757); 4 columns per thread (11 warps, the
// same time); a block barrier per plane (the same); one warp issuing all boxes
// (the others wait for it: 1000).
//
// Every wait is bounded and records DERR_TIMEOUT; a warp that gave up still takes
// part in every barrier of the plane loop, and the block waits for the copies it
// issued before it exits.
#include "evc_internal.cuh"
#include "evc_bulk.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <type_traits>

namespace evc {
namespace {

// Two columns in a 64-bit register: the packed FP32 instructions take half the
// issue slots, and every operation is rounded where it stands.
typedef unsigned long long F2;
__device__ __forceinline__ F2 add2(F2 a, F2 b)
{
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ F2 lds(uint32_t addr, int off)
{
    F2 d;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(d) : "r"(addr + off) : "memory");
    return d;
}
__device__ __forceinline__ void sts(uint32_t addr, int off, F2 v)
{
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(addr + off), "l"(v) : "memory");
}
__device__ __forceinline__ F2 pair2(float lo, float hi)
{
    F2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

constexpr int NC = 16;                   // columns of a block
constexpr int LPP = NC / 2;              // lanes per point
constexpr int NG = CW / NC;              // blocks per chunk and tile
constexpr int LA = 4;                    // planes of x in the ring
constexpr int UBUF = 4;                  // planes of u

template <int TS>
struct Geo {
    static constexpr int H = TS / 2;                 // points of one parity per row
    static constexpr int PP = H + 1;                 // patches per side of the tile with its ring
    static constexpr int NPATCH = PP * PP;
    static constexpr int NCW = (NPATCH * LPP + 31) / 32;   // consumer warps
    static constexpr int THREADS = NCW * 32;
    // one plane of x in points, every box on a 128-byte boundary: the tile by
    // parity [2][TS][H], the two columns left and right of it [TS][2], the two
    // rows below and above by parity [2][H], the corners' diagonal neighbours
    static constexpr int round(int pts) { return (pts * NC * 4 + 127) / 128 * 128 / (NC * 4); }
    static constexpr int PSTEP = round(TS * H), XSTEP = round(2 * TS), YSTEP = round(2 * H), CSTEP = round(1);
    static constexpr int X0 = 2 * PSTEP, Y0 = X0 + 2 * XSTEP, C0 = Y0 + 4 * YSTEP;
    static constexpr int PTS = C0 + 4 * CSTEP;
    static constexpr int BOXES = 2 + 2 + 4 + 4;
    static_assert(BOXES <= NCW, "a warp issues at most one box of a plane");
    // one plane of u by parity [TS + 2][2][PP]; a patch on the rim also reads one
    // row or point before or after it, for u values that nobody uses: the memory
    // there is the ring's, another plane's or the pad's
    static constexpr int UROW = PP, UPTS = round((TS + 2) * 2 * PP);
    static constexpr int XB = PTS * NC * 4, UB = UPTS * NC * 4;   // bytes of a plane
    static constexpr size_t SMEM = (size_t)LA * XB + (size_t)UBUF * UB + (2 * UROW + 2) * NC * 4;
};

struct PairArgs {
    int N, zb;
    // both halves the same: off-diagonal coefficient, each pass's scale and diagonal
    F2 c1, k1a, dga, k1b, dgb;
    F2 one;                  // 1: the second pass's scale of its stencil, rounded as there
    double a0;
    const double* insc;      // of x in the first pass, per column, or null
    const double* xs;        // of x in the last term, per column, or null
    const double* ppc;
    const void* pp;
    int64_t pp_cs;
    void* out;
    int64_t out_cs;
    const int* chunk_active;
    int* err;
    long long limit;         // clock cycles that a wait may take
    int have;                // planes whose first box is issued: all but in the self-test
};

// Maps over [chunk][y + N z][x / 2][x % 2][CW], by box (NC columns each): a
// tile's points of one parity, two columns, two rows of one parity, a point.
struct PairMaps {
    CUtensorMap box[4];
};

__device__ __forceinline__ void load5(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                      int c4, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
        "r"(smem_addr(bar))
        : "memory");
}

// Bounded wait that also gives up once the block's failure flag is set.
__device__ __forceinline__ bool wait_or(uint64_t* bar, uint32_t parity, volatile int* fail, long long limit)
{
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test(bar, parity)) {
        if (*fail) return false;
        if (clock64() - t0 > limit) {
            *fail = 1;
            return false;
        }
    }
    return true;
}

template <int TS, bool PP_>
__global__ void __launch_bounds__(Geo<TS>::THREADS, 1)
stencil_pair_kernel(const __grid_constant__ PairMaps maps, const PairArgs a)
{
    typedef Geo<TS> G;
    constexpr int NCW = G::NCW;
    const int ch = blockIdx.z;
    if (!a.chunk_active[ch]) return;
    extern __shared__ __align__(128) unsigned char raw[];
    if (smem_addr(raw) & 127) {
        if (threadIdx.x == 0) atomicExch(a.err, DERR_BOUNDS);
        return;
    }
    // planes of x [LA][PTS][NC], then of u [2][UPTS][NC]
    const uint32_t xbase = smem_addr(raw), ubase = xbase + LA * G::XB;
    __shared__ uint64_t full[LA];            // a plane of x has landed
    __shared__ uint64_t udone[2];            // every warp has stored its u of a plane (and read x for it)
    __shared__ int s_fail, s_last[G::BOXES];   // ... and the last plane that a box was issued of
    __shared__ int4 boxes[G::BOXES];
    if (threadIdx.x == 0) {
        for (int s = 0; s < LA; ++s) mbar_init(&full[s], G::BOXES);
        for (int s = 0; s < 2; ++s) mbar_init(&udone[s], NCW);
        s_fail = 0;
        for (int b = 0; b < G::BOXES; ++b) s_last[b] = -1;
        mbar_init_fence();
    }
    const int N = a.N;
    const int warp = threadIdx.x >> 5, l32 = threadIdx.x & 31;
    const int grp = blockIdx.x % NG, tile = blockIdx.x / NG;
    const int tiles = (N + TS - 1) / TS;
    // the last tile of a line that TS does not divide starts earlier: its points
    // that another tile also has get the same values from both
    const int x0 = min((tile % tiles) * TS, N - TS), y0 = min((tile / tiles) * TS, N - TS);
    const int z0 = blockIdx.y * a.zb, z1 = min(z0 + a.zb, N), nz = z1 - z0;
    volatile int* fail = &s_fail;
    auto wrap = [&](int v) { return v < 0 ? v + N : v >= N ? v - N : v; };
    const int nplane = nz + 4;               // x planes z0 - 2 .. z1 + 1

    // The boxes of a plane: {map, x, y, position in the stage}.  The two rows or
    // columns of an arm are even-aligned (N, x0 and y0 are even), so they wrap
    // together.  Box b of plane t (z0 - 2 + t) is issued by warp b, which alone
    // announces its bytes: a plane that some warps no longer issue, because a wait
    // gave up meanwhile, can still be waited for (below).
    if (threadIdx.x < G::BOXES) {
        const int b = threadIdx.x;
        int4 e;
        if (b < 2) e = make_int4(0, x0 + b, y0, b * G::PSTEP);
        else if (b < 4) e = make_int4(1, wrap(b == 2 ? x0 - 2 : x0 + TS), y0, G::X0 + (b - 2) * G::XSTEP);
        else if (b < 8) e = make_int4(2, x0 + (b & 1), wrap(b < 6 ? y0 - 2 : y0 + TS), G::Y0 + (b - 4) * G::YSTEP);
        else e = make_int4(3, wrap(b & 1 ? x0 + TS : x0 - 1), wrap(b & 2 ? y0 + TS : y0 - 1), G::C0 + (b - 8) * G::CSTEP);
        boxes[b] = e;
    }
    __syncthreads();
    const int pts = warp < 2 ? TS * G::H : warp < 4 ? 2 * TS : warp < 8 ? 2 * G::H : 1;    // of this warp's box
    auto issue = [&](int t, int stage) {
        if (warp >= G::BOXES || t >= nplane || l32 != 0 || *fail || (t >= a.have && warp == 0)) return;
        uint64_t* bar = &full[stage];
        int z = z0 - 2 + t;
        z = z < 0 ? z + N : z >= N ? z - N : z;
        const int4 e = boxes[warp];
        mbar_arrive_expect_tx(bar, pts * NC * 4);
        load5(xbase + stage * G::XB + e.w * NC * 4, &maps.box[e.x], grp * NC, e.y & 1, e.y >> 1, z * N + e.z, ch, bar);
        s_last[warp] = t;
    };
#pragma unroll
    for (int t = 0; t < LA; ++t) issue(t, t);
    {
        const int sub = threadIdx.x % LPP, patch = min((int)threadIdx.x / LPP, G::NPATCH - 1);
        const bool live = (int)threadIdx.x / LPP < G::NPATCH;
        const int px = patch % G::PP, py = patch / G::PP;
        const int ex = 2 * px - 1, ey = 2 * py - 1;      // the patch's first point, tile coordinates
        // position of tile point (tx, ty) in a staged plane (points outside the
        // diamond are read only for u values nobody uses)
        auto at = [&](int tx, int ty) {
            const bool ix = tx >= 0 && tx < TS, iy = ty >= 0 && ty < TS;
            const int ax = tx < 0 ? tx + 2 : tx - TS + 2, ay = ty < 0 ? ty + 2 : ty - TS + 2;
            int p = 0;
            if (ix && iy) p = (tx & 1) * G::PSTEP + ty * G::H + (tx >> 1);
            else if (iy) p = G::X0 + (ax >> 1) * G::XSTEP + ty * 2 + (ax & 1);
            else if (ix) p = G::Y0 + ((ay >> 1) * 2 + (tx & 1)) * G::YSTEP + (ay & 1) * G::H + (tx >> 1);
            else if ((ax == 1 || ax == 2) && (ay == 1 || ay == 2)) p = G::C0 + ((ax == 2 ? 1 : 0) + (ay == 2 ? 2 : 0)) * G::CSTEP;
            return xbase + (uint32_t)(p * NC * 4 + sub * 8);
        };
        uint32_t own[4], hl[2], hr[2], hd[2], hu[2];          // own points; left, right, below, above
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            own[2 * b] = at(ex, ey + b);
            own[2 * b + 1] = at(ex + 1, ey + b);
            hl[b] = at(ex - 1, ey + b);
            hr[b] = at(ex + 2, ey + b);
            hd[b] = at(ex + b, ey - 1);
            hu[b] = at(ex + b, ey + 2);
        }
        // u plane: point (ex + qx, ey + qy), qx and qy in -1 .. 2
        const uint32_t u0 = ubase + ((2 * py * 2 * G::UROW + px) * NC * 4 + sub * 8);
        auto uat = [](int qx, int qy) {
            return (qy * 2 * G::UROW + (qx & 1) * G::UROW + (qx < 0 ? -1 : qx >> 1)) * NC * 4;
        };
        const int cc = grp * NC + sub * 2;               // first column within the chunk
        const int c = ch * CW + cc;
        const F2 insc = a.insc ? pair2((float)a.insc[c], (float)a.insc[c + 1]) : pair2(1.0f, 1.0f);
        const F2 a0c = pair2((float)(a.a0 * (a.xs ? a.xs[c] : 1.0)), (float)(a.a0 * (a.xs ? a.xs[c + 1] : 1.0)));
        const F2 nppc = PP_ ? pair2(-(float)a.ppc[c], -(float)a.ppc[c + 1]) : 0;
        const int64_t NN = (int64_t)N * N;
        // output points: offset of the first one, and which of the four are the tile's
        const int g0 = (x0 + ex) + N * (y0 + ey);
        unsigned mine = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int tx = ex + (q & 1), ty = ey + (q >> 1);
            if (live && tx >= 0 && tx < TS && ty >= 0 && ty < TS) mine |= 1u << q;
        }
        auto gpt = [&](int q, int64_t plane) { return (plane + g0 + (q & 1) + (q >> 1) * N) * CW; };
        float* out = static_cast<float*>(a.out) + ch * a.out_cs + cc;
        const float* pp = PP_ ? static_cast<const float*>(a.pp) + ch * a.pp_cs + cc : nullptr;
        // c1 (xl + xr + yl + yr + zl + zr), then k1 times it plus dg x, as the single pass
        auto stencil = [&](F2 xl, F2 xr, F2 yl, F2 yr, F2 zl, F2 zr, F2 x, F2 k1, F2 dg) {
            const F2 off = mul2(a.c1, add2(add2(add2(add2(add2(xl, xr), yl), yr), zl), zr));
            return fma2(k1, off, mul2(dg, x));
        };

        F2 xw[3][4], uw[3][4];
        bool ok = true;
        auto take = [&](int stage, uint32_t parity, F2* x) {        // own points of a plane
            ok = ok && __all_sync(0xffffffffu, wait_or(&full[stage], parity, fail, a.limit));
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = lds(own[q], stage * G::XB);
        };
        take(0, 0, xw[0]);
        take(1, 0, xw[1]);
        int64_t plane = NN * (z0 - 2);                   // of out in step j
        // step j: u of plane z0 - 1 + j (x planes t = j, j + 1, j + 2 of the ring),
        // out of plane z0 - 2 + j.  S = j % LA fixes the ring stages and the
        // places in the windows; round = j / LA.
        auto step = [&](auto S, int j, uint32_t round) {
            constexpr int s = decltype(S)::value;
            F2 *xm = xw[s % 3], *xc = xw[(s + 1) % 3], *xp = xw[(s + 2) % 3];
            F2 *um = uw[(s + 1) % 3], *uc = uw[(s + 2) % 3], *up = uw[s % 3];
            constexpr int xo = (s + 1) % LA * G::XB, un = s % UBUF * G::UB, us = (s + UBUF - 1) % UBUF * G::UB;
            take((s + 2) % LA, (round + (s + 2) / LA) & 1, xp);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const F2 l = lds(hl[b], xo), r = lds(hr[b], xo);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int p = 2 * b + q;
                    const F2 o = lds(b ? hu[q] : hd[q], xo);
                    up[p] = mul2(insc, stencil(q ? xc[p - 1] : l, q ? r : xc[p + 1], b ? xc[q] : o, b ? o : xc[2 + q],
                                               xm[p], xp[p], xc[p], a.k1a, a.dga));
                    if (live) sts(u0, un + uat(q, b), up[p]);
                }
            }
            // (No proxy fence before the stage of plane j is refilled, as the reorthogonalisation
            // kernels have: every value read from it has gone into a u stored above, so the
            // reads are complete.  A read whose value is used later would need one: 1 % of a
            // Chebyshev count.)
            __syncwarp();
            if (l32 == 0) mbar_arrive(&udone[s & 1]);
            if (j >= 1) {
                // every warp is done with plane j - 1 of u, hence with plane j of x,
                // whose stage takes the next plane to load
                ok = ok && __all_sync(0xffffffffu, wait_or(&udone[(s + 1) & 1], ((j - 1) >> 1) & 1, fail, a.limit));
                if (j == 1) issue(LA, 0);
                issue(j + LA, s % LA);
            }
            if (j >= 2) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const F2 l = lds(u0, us + uat(-1, b)), r = lds(u0, us + uat(2, b));
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int p = 2 * b + q;
                        const F2 o = lds(u0, us + uat(q, b ? 2 : -1));
                        const F2 sv = stencil(q ? uc[p - 1] : l, q ? r : uc[p + 1], b ? uc[q] : o, b ? o : uc[2 + q],
                                              um[p], up[p], uc[p], a.k1b, a.dgb);
                        F2 res = fma2(a.one, sv, mul2(a0c, xm[p]));
                        if (mine >> p & 1) {
                            if (PP_) res = fma2(nppc, *reinterpret_cast<const F2*>(pp + gpt(p, plane)), res);
                            *reinterpret_cast<F2*>(out + gpt(p, plane)) = res;
                        }
                    }
                }
            }
            plane += NN;
        };
        static_assert(LA == 4 && UBUF == 4, "twelve steps are unrolled: windows of 3, 4 planes of u and of x");
        const int J = nz + 2;
        for (int jb = 0, round = 0; jb < J; jb += 12, round += 12 / LA) {
            step(std::integral_constant<int, 0>(), jb, round);
            if (jb + 1 < J) step(std::integral_constant<int, 1>(), jb + 1, round);
            if (jb + 2 < J) step(std::integral_constant<int, 2>(), jb + 2, round);
            if (jb + 3 < J) step(std::integral_constant<int, 3>(), jb + 3, round);
            if (jb + 4 < J) step(std::integral_constant<int, 4>(), jb + 4, round);
            if (jb + 5 < J) step(std::integral_constant<int, 5>(), jb + 5, round);
            if (jb + 6 < J) step(std::integral_constant<int, 6>(), jb + 6, round);
            if (jb + 7 < J) step(std::integral_constant<int, 7>(), jb + 7, round);
            if (jb + 8 < J) step(std::integral_constant<int, 8>(), jb + 8, round);
            if (jb + 9 < J) step(std::integral_constant<int, 9>(), jb + 9, round);
            if (jb + 10 < J) step(std::integral_constant<int, 10>(), jb + 10, round);
            if (jb + 11 < J) step(std::integral_constant<int, 11>(), jb + 11, round);
        }
    }
    __syncthreads();
    // Every plane issued was waited for, unless a wait gave up.  Then, before the
    // shared memory is released: arrive in the place of the warps that issued no box
    // of a plane any more, and wait (again with the limit) for the others' boxes.  A
    // plane was issued only once every warp had seen the one before it in its stage,
    // so the last LA planes are the ones that can be in flight.
    if (*fail) {
        if (threadIdx.x == 0) {
            atomicCAS(a.err, DERR_NONE, DERR_TIMEOUT);
            int most = -1;
            for (int b = 0; b < G::BOXES; ++b) most = max(most, s_last[b]);
            for (int t = max(0, most - LA + 1); t <= most; ++t) {
                for (int b = 0; b < G::BOXES; ++b)
                    if (s_last[b] < t) mbar_arrive(&full[t % LA]);
                mbar_wait_for(&full[t % LA], (t / LA) & 1, a.limit);
            }
        }
    }
    __syncthreads();
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        return PFN_cuTensorMapEncodeTiled_v12000(nullptr);
    }();
    return fn;
}

bool encode(CUtensorMap* m, const void* base, int64_t cs, int N, int cn, int bpar, int bxh, int by)
{
    auto fn = encode_fn();
    if (!fn || !base) return false;
    const cuuint64_t pt = CW * sizeof(float);
    cuuint64_t dim[5] = {(cuuint64_t)CW, 2, (cuuint64_t)(N / 2), (cuuint64_t)N * N, (cuuint64_t)cn};
    cuuint64_t str[4] = {pt, 2 * pt, pt * N, (cuuint64_t)cs * sizeof(float)};
    cuuint32_t box[5] = {(cuuint32_t)NC, (cuuint32_t)bpar, (cuuint32_t)bxh, (cuuint32_t)by, 1};
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<void*>(base), dim, str, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int TS, bool PP_>
cudaError_t launch(dim3 grid, cudaStream_t st, const PairMaps& m, const PairArgs& a)
{
    static std::atomic<uint64_t> attr{0};
    const cudaError_t e = smem_limit_once(attr, stencil_pair_kernel<TS, PP_>, Geo<TS>::SMEM);
    if (e != cudaSuccess) return e;
    stencil_pair_kernel<TS, PP_><<<grid, Geo<TS>::THREADS, Geo<TS>::SMEM, st>>>(m, a);
    return cudaGetLastError();
}

// Tile side and z planes per block (at most the caller's zb).  A block takes one
// SM, marches its planes and recomputes about 3.5 more at its ends; a plane's time
// goes with the patches of the tile and its ring: the choice with the smallest
// (waves of blocks) x (planes + 3.5) x ((TS + 2)^2 / 4 + 10).  16 where it divides
// N; 14 or 12 where they cover N with fewer points (N = 40, 56, 72).
struct Shape {
    int ts, zb;
};
Shape choose_shape(int N, int nchunk, int zb)
{
    double best = 1e300;
    Shape r{16, N};
    for (int ts : {16, 14, 12}) {
        if (ts > N) continue;
        const int tiles = (N + ts - 1) / ts, smax = (N + 3) / 4;
        const int64_t per = (int64_t)tiles * tiles * NG * nchunk;     // blocks per segment
        for (int s = 1; s <= smax; ++s) {
            const int z = (N + s - 1) / s;
            if (z > zb && s < smax) continue;
            const double cost = (double)((per * s + 151) / 152) * (z + 3.5) * ((ts + 2) * (ts + 2) / 4 + 10);
            if (cost < best) {
                best = cost;
                r = Shape{ts, z};
            }
        }
    }
    return r;
}

template <int TS>
cudaError_t launch_ts(const StencilOp& op, const StencilPass& p, const PairArgs& a, int cn, cudaStream_t st)
{
    const int N = op.N;
    PairMaps m;
    std::memset(&m, 0, sizeof m);
    if (!encode(&m.box[0], p.in, p.in_cs, N, cn, 1, TS / 2, TS) || !encode(&m.box[1], p.in, p.in_cs, N, cn, 2, 1, TS) ||
        !encode(&m.box[2], p.in, p.in_cs, N, cn, 1, TS / 2, 2) || !encode(&m.box[3], p.in, p.in_cs, N, cn, 1, 1, 1))
        return cudaErrorInvalidValue;
    const int tiles = (N + TS - 1) / TS;
    dim3 grid((unsigned)(tiles * tiles * NG), (unsigned)((N + a.zb - 1) / a.zb), (unsigned)cn);
    return p.pp ? launch<TS, true>(grid, st, m, a) : launch<TS, false>(grid, st, m, a);
}

}  // namespace

// FP32 7-point passes on grids with N even and at least the smallest tile.  Not for
// many columns on grids of little more than a tile, which the tiles cover one and a
// half to two times, where the single passes run on patches that march whole lines or
// overlap in chunk groups.  ms of 6 steps, 2 x 2 patches, pair | single passes: 32
// chunks, 4 groups, 16 z planes per block N = 18 2.74 | 2.50, 20 2.98 | 2.72, 22 3.38 |
// 3.15; 64 chunks, one group N = 18 5.40 | 4.67, 20 6.01 | 5.36, 22 6.89 | 6.25.  At N = 24
// (two tiles, exactly) with 32 chunks it is 3.51 | 4.23, and from N = 26 on, or with less
// work than this, the pair is faster too (N = 22, 16 chunks, 4 steps 0.88 | 0.93).
bool stencil_pair_eligible(const StencilOp& op, size_t tsize, int nchunk)
{
    if (tsize != 4 || op.order != 2 || op.N < 12 || op.N % 2 || encode_fn() == nullptr) return false;
    const bool patches = op.patch >= 2 && (op.cn > 0 || (op.zb > 0 ? op.zb : 32) >= op.N);
    return !(patches && op.N > 16 && op.N < 24 && (int64_t)op.N * op.N * op.N * nchunk >= 180000);
}

// first: x -> u (in, insc, k1, k0); second: u -> out (k1, k0, x, xs, a0, pp, ppc, out).
cudaError_t launch_stencil_pair(const StencilOp& op, const Run& r, const StencilPass& first,
                                const StencilPass& second, cudaStream_t st)
{
    const int c0 = op.cn > 0 ? op.c0 : 0, cn = op.cn > 0 ? op.cn : r.nchunk;
    if (c0 < 0 || c0 + cn > r.nchunk || !stencil_pair_eligible(op, 4, r.nchunk)) return cudaErrorInvalidValue;
    if (first.in != second.x || first.in_cs != second.x_cs || first.in == second.out || first.useV ||
        second.useV || second.prev || first.pp || first.x)
        return cudaErrorInvalidValue;
    auto at = [&](const void* q, int64_t cs) { return static_cast<const float*>(q) + (int64_t)c0 * cs; };
    auto atc = [&](const double* q) { return q ? q + (int64_t)c0 * CW : q; };
    StencilPass p = first;
    p.in = at(first.in, first.in_cs);
    p.pp = second.pp;
    PairArgs a{};
    a.N = op.N;
    auto both = [](double v) {
        const float f = (float)v;
        uint32_t b;
        std::memcpy(&b, &f, 4);
        return (F2)b << 32 | b;
    };
    a.c1 = both(op.c1);
    a.k1a = both(first.k1);
    a.dga = both(std::fma(first.k1, op.cd, first.k0));
    a.k1b = both(second.k1);
    a.dgb = both(std::fma(second.k1, op.cd, second.k0));
    a.one = both(1.0);
    a.a0 = second.a0;
    a.insc = atc(first.insc);
    a.xs = atc(second.xs);
    a.ppc = atc(second.ppc);
    a.pp = second.pp ? at(second.pp, second.pp_cs) : nullptr;
    a.pp_cs = second.pp_cs;
    a.out = const_cast<float*>(at(second.out, second.out_cs));
    a.out_cs = second.out_cs;
    a.chunk_active = r.chunk_active + c0;
    a.err = r.err;
    a.limit = kWaitCycles;
    a.have = INT_MAX;
    const Shape sh = choose_shape(op.N, r.nchunk, op.zb > 0 ? op.zb : 64);
    a.zb = sh.zb;
    return sh.ts == 16   ? launch_ts<16>(op, p, a, cn, st)
           : sh.ts == 14 ? launch_ts<14>(op, p, a, cn, st)
                         : launch_ts<12>(op, p, a, cn, st);
}

// The failure path on a 12^3 grid: plane 2 lacks its first box, so the waits for it
// give up after `cycles` and the block winds down with the plane's other boxes in
// flight.  *err (device memory) receives DERR_TIMEOUT.
cudaError_t stencil_pair_selftest(long long cycles, int* err)
{
    constexpr int N = 12;
    const size_t vec = (size_t)N * N * N * CW;
    float* buf = nullptr;                        // x, out, then a chunk's flag
    cudaError_t e = cudaMalloc(&buf, (2 * vec + 1) * sizeof(float));
    if (e != cudaSuccess) return e;
    PairArgs a{};
    a.N = N;
    a.zb = N;
    a.out = buf + vec;
    a.out_cs = (int64_t)vec;
    int* active = reinterpret_cast<int*>(buf + 2 * vec);
    a.chunk_active = active;
    a.err = err;
    a.limit = cycles;
    a.have = 2;
    StencilOp op{};
    op.N = N;
    StencilPass p{};
    p.in = buf;
    p.in_cs = (int64_t)vec;
    const int one = 1;
    e = cudaMemset(buf, 0, 2 * vec * sizeof(float));
    if (e == cudaSuccess) e = cudaMemcpy(active, &one, sizeof one, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = launch_ts<12>(op, p, a, 1, nullptr);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(buf);
    return e;
}

}  // namespace evc
