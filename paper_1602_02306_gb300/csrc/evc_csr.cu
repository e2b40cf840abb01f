// evc_csr.cu -- the preconditioned shifted operator for a CSR matrix,
//   w = M (A - sigma_c I) M q_i - beta_i q_{i-1}       (Algorithm 1, first
// line of the loop body), with M = I or the Jacobi scaling
// M = diag((|a_rr - sigma| + eps)^(-1/2)) fused as row and column scales;
// or, for the T^{-1}-inner-product process (Sec. 4, Eq. lanT1) with T = M^2,
//   w = T (A - sigma_c I) y_i - beta_i y_{i-1},
// where T is a row scale only and the gathered rows are not scaled.
//
// Row r of C x is  m_r sum_{j != r} a_rj m_j x_j  +  d_r x_r  with the
// diagonal d_r = (a_rr - sigma) m_r^2 (or a_rr - sigma without M) taken from
// a per-shift array formed in FP64: the stored diagonal entries are skipped in
// the row sum, so in FP32 the shift never cancels against a_rr, and a rounded
// a_rr never reaches m_r^2, which magnifies it by up to 1/eps.
//
// Every gathered x row of a chunk is one contiguous 128-byte (FP32) / 256-byte
// (FP64) segment; q_i = s_i P_i is scaled on the fly.
#include "evc_internal.cuh"

#include <cstring>
#include <type_traits>

namespace evc {
namespace {

struct CArgs {
    CsrOp op;
    const void* x;          // slot i-1 of the basis (P_i)
    const void* gx;         // its scaled copy m_r x_r (gather_copy), or null
    const void* pp;         // slot i-2 (P_{i-1}) or null
    void* out;              // slot i
    int64_t chunk_stride;
    const double* insc;     // s_i per column
    const double* ppc;      // beta_i s_{i-1} per column
    const int* shift_of;
    const void* jac;
    const void* dsh;        // T[S][n] diagonal of the shifted (scaled) operator
    const int* chunk_active;
};

template <typename T> struct alignas(16) Pack { T v[16 / sizeof(T)]; };
template <typename T> struct Vec16;
template <> struct Vec16<float> { typedef float4 type; };
template <> struct Vec16<double> { typedef double2 type; };

// Row sums are accumulated entry by entry, acc = fma(a_rj, x_j m_j, acc), with
// the product and the fused multiply-add rounded explicitly, so that every
// specialisation of the pass (uniform-shift chunks or not, any block size)
// gives bitwise the same rows: a column's result must not depend on which
// kernel its batch ran.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename T>
__device__ __forceinline__ Pack<T> ldg16(const T* p)
{
    typename Vec16<T>::type t = __ldg(reinterpret_cast<const typename Vec16<T>::type*>(p));
    Pack<T> r;
    memcpy(&r, &t, 16);
    return r;
}

// L2 policy of data that a pass reads or writes once: first to be evicted, so
// that it does not push out the x rows, which are gathered again and again.
__device__ __forceinline__ uint64_t policy_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ int ld_once(const int* p, uint64_t pol)
{
    int v;
    asm volatile("ld.global.nc.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_once(const float* p, uint64_t pol)
{
    float v;
    asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ double ld_once(const double* p, uint64_t pol)
{
    double v;
    asm volatile("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
    return v;
}
template <typename T>
__device__ __forceinline__ Pack<T> ld_once(const Pack<T>* p, uint64_t pol)
{
    uint4 t;
    asm volatile("ld.global.nc.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(t.x), "=r"(t.y), "=r"(t.z), "=r"(t.w) : "l"(p), "l"(pol));
    Pack<T> r;
    memcpy(&r, &t, 16);
    return r;
}
template <typename T>
__device__ __forceinline__ void st_once(Pack<T>* p, const Pack<T>& v, uint64_t pol)
{
    uint4 t;
    memcpy(&t, &v, 16);
    asm volatile("st.global.L2::cache_hint.v4.b32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(t.x),
                 "r"(t.y), "r"(t.z), "r"(t.w), "l"(pol)
                 : "memory");
}

// A group of LPR = CW / W lanes owns one row of one chunk; each lane holds W
// consecutive columns (one 16-byte vector), so one gather instruction of the
// warp fetches 32/LPR whole x rows.  Rows are visited in the order of
// op.perm (rows sorted by length, longest first) so the rows sharing a warp
// have similar lengths; each group broadcasts the row's (col, val) pairs from
// its own lanes with warp shuffles.  UNI: every chunk's 32 columns belong to
// one shift (m a multiple of 32, or one shift), so a gathered entry needs one
// Jacobi scale, not one per column.  This kernel is the pass that scales the
// gathered rows (PM_JACOBI without a scaled copy); csr_gather_kernel the others.
template <typename T, bool UNI, int NT>
__global__ void __launch_bounds__(NT)
csr_pass_kernel(CArgs a)
{
    constexpr int W = 16 / sizeof(T);
    constexpr int LPR = CW / W;                 // lanes per row
    constexpr int RPW = 32 / LPR;               // rows per warp
    const int ch = blockIdx.y;
    if (!a.chunk_active[ch]) return;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int64_t slotrow = ((int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5)) * RPW + grp;
    const int64_t n = a.op.n;
    const bool valid = slotrow < n;
    const int64_t row = valid ? (a.op.perm ? (int64_t)a.op.perm[slotrow] : slotrow) : 0;
    const int c0 = ch * CW + sub * W;
    const T* x = static_cast<const T*>(a.x) + ch * a.chunk_stride;
    const T* val = static_cast<const T*>(a.op.val);
    constexpr int NJ = UNI ? 1 : W;             // Jacobi scale arrays in use
    const T* jr[NJ];
#pragma unroll
    for (int w = 0; w < NJ; ++w)
        jr[w] = static_cast<const T*>(a.jac) + (int64_t)a.shift_of[c0 + w] * n;

    const int64_t beg = valid ? a.op.row_ptr[row] : 0, end = valid ? a.op.row_ptr[row + 1] : 0;
    // the warp walks the longest of its rows; shorter rows contribute zeros
    int64_t len = end - beg, mx = len;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, (int64_t)__shfl_xor_sync(0xffffffffu, mx, o));
    T acc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) acc[w] = 0;
    for (int64_t k0 = 0; k0 < mx; k0 += LPR) {
        const int64_t kk = beg + k0 + sub;
        int mycol = (int)row;
        T myval = 0;
        if (k0 + sub < len) {
            mycol = __ldg(a.op.col + kk);
            myval = mycol == (int)row ? (T)0 : __ldg(val + kk);   // diagonal: from dsh
        }
        const int cnt = (int)min((int64_t)LPR, mx - k0);
        int t = 0;
        for (; t + 1 < cnt; t += 2) {
            const int ca = __shfl_sync(0xffffffffu, mycol, grp * LPR + t);
            const int cb = __shfl_sync(0xffffffffu, mycol, grp * LPR + t + 1);
            const T va = __shfl_sync(0xffffffffu, myval, grp * LPR + t);
            const T vb = __shfl_sync(0xffffffffu, myval, grp * LPR + t + 1);
            Pack<T> xa = ldg16(x + (int64_t)ca * CW + sub * W);
            Pack<T> xb = ldg16(x + (int64_t)cb * CW + sub * W);
            T ma = 1, mb = 1;
            if (UNI) { ma = __ldg(jr[0] + ca); mb = __ldg(jr[0] + cb); }
#pragma unroll
            for (int w = 0; w < W; ++w) {
                T sa = xa.v[w], sb = xb.v[w];
                if (UNI) { sa = mul_rn(sa, ma); sb = mul_rn(sb, mb); }
                if (!UNI) {
                    sa = mul_rn(sa, __ldg(jr[w] + ca));
                    sb = mul_rn(sb, __ldg(jr[w] + cb));
                }
                acc[w] = fma_rn(vb, sb, fma_rn(va, sa, acc[w]));
            }
        }
        if (t < cnt) {
            const int ca = __shfl_sync(0xffffffffu, mycol, grp * LPR + t);
            const T va = __shfl_sync(0xffffffffu, myval, grp * LPR + t);
            Pack<T> xa = ldg16(x + (int64_t)ca * CW + sub * W);
            const T ma = UNI ? __ldg(jr[0] + ca) : (T)1;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                T sa = xa.v[w];
                if (UNI) sa = mul_rn(sa, ma);
                if (!UNI) sa = mul_rn(sa, __ldg(jr[w] + ca));
                acc[w] = fma_rn(va, sa, acc[w]);
            }
        }
    }
    if (!valid) return;
    const Pack<T> cen = ldg16(x + row * CW + sub * W);
    const T* pp = a.pp ? static_cast<const T*>(a.pp) + ch * a.chunk_stride : nullptr;
    Pack<T> prev;
    if (pp) prev = ldg16(pp + row * CW + sub * W);
    const T* dsh = static_cast<const T*>(a.dsh);
    Pack<T> res;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int c = c0 + w;
        T r = acc[w];
        r = mul_rn(r, __ldg(jr[UNI ? 0 : w] + row));
        r = fma_rn(__ldg(dsh + (int64_t)a.shift_of[c] * n + row), cen.v[w], r);
        r = mul_rn(r, (T)a.insc[c]);
        if (pp) r = fma_rn(-(T)a.ppc[c], prev.v[w], r);
        res.v[w] = r;
    }
    typename Vec16<T>::type o;
    memcpy(&o, &res, 16);
    *reinterpret_cast<typename Vec16<T>::type*>(static_cast<T*>(a.out) + ch * a.chunk_stride +
                                                  row * CW + sub * W) = o;
}

// The pass on rows gathered as they are: PM_NONE, PM_TLEFT (output rows scaled
// by T = m^2, which jac then holds) and, with PRE, PM_JACOBI from the scaled copy
// of q_i.  Same ownership, same order of the sums and same roundings as above.
// Bound by the latency of the gathers (128 or 256 bytes at random from L2 and
// DRAM): all eight of a batch are in flight, the next batch of (col, val) pairs
// is fetched meanwhile, and what the pass touches once leaves L2 first.  The bound
// on the registers (56 and 36 warps per SM with 128 threads, 64 and 32 with 256 and
// 512, whose blocks come in fours and twos) holds the batch (two gathers in flight:
// 30 % slower; eight without the bound: 1.18, 1.51 and 1.73 ms with 128, 64 and 256
// threads; with it 1.01 and 1.06 with 128 and 256).
// FP32 rows are padded to whole batches (their own row of x, times zero): smaller
// batches for the rest cost more than the gathers they save (2M rows, six passes:
// 25.5 | 26.2 to 27.0 ms).  FP64 rows are not: a padded entry takes the FP64 units,
// which bound the pass, as long as a real one (500k rows of 3, 5, 7 and 13 entries,
// six passes: 3.7, 3.7, 3.7, 6.5 | 2.4, 2.9, 3.4, 5.4 ms).  ms per pass, before | now:
//   64 columns x 2 shifts, power-law rows (mean 29), FP32, T^-1 process: 600k
//   rows 1.44 | 1.00, 2M 4.85 | 4.41; Jacobi: 2M 5.28 | 4.60 and 0.16 more in the
//   kernel that writes the copy, 600k 1.66 | 1.10, 30k (one row of 2000 entries
//   is the critical path) 0.55 | 0.21; FP64 Jacobi 200k 2.49 | 1.42 (FP64 units:
//   one operation per entry and column, before two).
// 2M rows move 6.8 GB per chunk through DRAM (the 256 MB of a chunk's x are twice L2)
// at 6.25 TB/s, 0.92 of the copy peak: hits in L2 not counted, which make it 7.2.  Slices of 16 or 8 columns of x, which fit L2, are no way out: 64
// and 32-byte gathers took 6.5 and 10.7 ms per pass.
template <typename T, int PM, int NT, bool PRE>
__global__ void __launch_bounds__(NT, 36 * 32 / NT)
csr_gather_kernel(CArgs a)
{
    static_assert(PM != PM_JACOBI || PRE, "the gathered rows are not scaled here");
    constexpr int W = 16 / sizeof(T);
    constexpr int LPR = CW / W;
    constexpr int RPW = 32 / LPR;
    constexpr int U = 8;                        // gathers in flight per lane
    const int ch = blockIdx.y;
    if (!a.chunk_active[ch]) return;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int64_t slotrow = ((int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5)) * RPW + grp;
    const int64_t n = a.op.n;
    const bool valid = slotrow < n;
    const int64_t row = valid ? (a.op.perm ? (int64_t)a.op.perm[slotrow] : slotrow) : 0;
    const T* y = static_cast<const T*>(PRE ? a.gx : a.x) + ch * a.chunk_stride + sub * W;
    const int64_t beg = valid ? a.op.row_ptr[row] : 0, len = valid ? a.op.row_ptr[row + 1] - beg : 0;
    int64_t mx = len;
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1) mx = max(mx, (int64_t)__shfl_xor_sync(0xffffffffu, mx, o));
    const uint64_t once = policy_first();
    const int32_t* col = a.op.col + beg;
    const T* val = static_cast<const T*>(a.op.val) + beg;
    T acc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) acc[w] = 0;
    int ncol = (int)row;
    T nval = 0;
    if (sub < len) {
        ncol = ld_once(col + sub, once);
        nval = ld_once(val + sub, once);
    }
    for (int64_t k0 = 0; k0 < mx; k0 += LPR) {
        const int mycol = ncol;
        const T myval = mycol == (int)row ? (T)0 : nval;       // diagonal: from dsh
        ncol = (int)row;
        nval = 0;
        if (k0 + LPR + sub < len) {
            ncol = ld_once(col + k0 + LPR + sub, once);
            nval = ld_once(val + k0 + LPR + sub, once);
        }
        const int cnt = (int)min((int64_t)LPR, mx - k0);
        auto batch = [&](auto size, int t) {
            constexpr int B = decltype(size)::value;
            Pack<T> xv[B];
#pragma unroll
            for (int u = 0; u < B; ++u)
                xv[u] = ldg16(y + (int64_t)__shfl_sync(0xffffffffu, mycol, grp * LPR + t + u) * CW);
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const T v = __shfl_sync(0xffffffffu, myval, grp * LPR + t + u);
#pragma unroll
                for (int w = 0; w < W; ++w) acc[w] = fma_rn(v, xv[u].v[w], acc[w]);
            }
        };
        if constexpr (sizeof(T) == 4) {
            static_assert(sizeof(T) == 8 || U == LPR, "one batch holds a row's lanes");
            batch(std::integral_constant<int, U>(), 0);
        } else {
            int t = 0;
            for (; t + U <= cnt; t += U) batch(std::integral_constant<int, U>(), t);
            if (cnt & 4) {
                batch(std::integral_constant<int, 4>(), t);
                t += 4;
            }
            if (cnt & 2) {
                batch(std::integral_constant<int, 2>(), t);
                t += 2;
            }
            if (cnt & 1) batch(std::integral_constant<int, 1>(), t);
        }
    }
    if (!valid) return;
    const int64_t at = ch * a.chunk_stride + row * CW + sub * W;
    const Pack<T> cen = ldg16(static_cast<const T*>(a.x) + at);
    Pack<T> prev, res;
    if (a.pp) prev = ld_once(reinterpret_cast<const Pack<T>*>(static_cast<const T*>(a.pp) + at), once);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int c = ch * CW + sub * W + w;
        const int64_t sr = (int64_t)a.shift_of[c] * n + row;
        T r = acc[w];
        if (PM != PM_NONE) r = mul_rn(r, __ldg(static_cast<const T*>(a.jac) + sr));
        r = fma_rn(__ldg(static_cast<const T*>(a.dsh) + sr), cen.v[w], r);
        r = mul_rn(r, (T)a.insc[c]);
        if (a.pp) r = fma_rn(-(T)a.ppc[c], prev.v[w], r);
        res.v[w] = r;
    }
    st_once(reinterpret_cast<Pack<T>*>(static_cast<T*>(a.out) + at), res, once);
}

}  // namespace

template <typename T>
cudaError_t launch_csr_pass(const CsrOp& op, const Run& r, int i, int pmode, cudaStream_t st)
{
    // step i reads slot i-1 (q_i), slot i-2 (q_{i-1}) and writes slot i
    CArgs a;
    a.op = op;
    T* basis = static_cast<T*>(r.basis);
    a.x = basis + (int64_t)(i - 1) * r.slot_stride;
    // the three-term term -beta_i q_{i-1} is Lanczos only
    a.pp = (i >= 2 && !r.arnoldi) ? basis + (int64_t)(i - 2) * r.slot_stride : nullptr;
    a.out = basis + (int64_t)i * r.slot_stride;
    a.chunk_stride = r.chunk_stride;
    a.insc = r.scl + (int64_t)(i - 1) * r.ncol;
    a.ppc = r.ppc;
    a.shift_of = r.shift_of;
    a.jac = r.jac;
    a.dsh = r.dsh;
    a.chunk_active = r.chunk_active;
    constexpr int RPW = 32 / (CW / (16 / (int)sizeof(T)));
    const int nt = op.threads > 0 ? op.threads : kThreads;
    const int rows_per_block = (nt / 32) * RPW;
    dim3 grid((unsigned)((op.n + rows_per_block - 1) / rows_per_block), r.nchunk);
    // every chunk's columns share one shift when m is a multiple of 32 (the
    // padding columns of the last chunk take the last shift) or S = 1
    const bool uni = r.S == 1 || r.m % CW == 0;
    a.gx = gather_copy(r, i) ? basis + (int64_t)(i + 1) * r.slot_stride : nullptr;
    auto launch = [&](auto nt_t) -> bool {
        constexpr int NT = decltype(nt_t)::value;
        if (pmode == PM_NONE) csr_gather_kernel<T, PM_NONE, NT, false><<<grid, NT, 0, st>>>(a);
        else if (pmode == PM_TLEFT) csr_gather_kernel<T, PM_TLEFT, NT, false><<<grid, NT, 0, st>>>(a);
        else if (pmode != PM_JACOBI) return false;
        else if (a.gx) csr_gather_kernel<T, PM_JACOBI, NT, true><<<grid, NT, 0, st>>>(a);
        else if (uni) csr_pass_kernel<T, true, NT><<<grid, NT, 0, st>>>(a);
        else csr_pass_kernel<T, false, NT><<<grid, NT, 0, st>>>(a);
        return true;
    };
    bool ok = false;
    switch (nt) {
    case 128: ok = launch(std::integral_constant<int, 128>()); break;
    case 256: ok = launch(std::integral_constant<int, 256>()); break;
    case 512: ok = launch(std::integral_constant<int, 512>()); break;
    }
    if (!ok) return cudaErrorInvalidValue;
    return cudaGetLastError();
}

template cudaError_t launch_csr_pass<float>(const CsrOp&, const Run&, int, int, cudaStream_t);
template cudaError_t launch_csr_pass<double>(const CsrOp&, const Run&, int, int, cudaStream_t);

}  // namespace evc
