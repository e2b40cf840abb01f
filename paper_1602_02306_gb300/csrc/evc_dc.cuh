// evc_dc.cuh -- eigenvalues and first eigenvector components of a symmetric
// tridiagonal J_k (the nodes and weights of Sec. 3, Eq. gauss_quad) by Cuppen's
// divide and conquer, one thread block per matrix or, for many short ones, several
// matrices per warp.  (Also compiled by the host compiler, which tests the phases.)
//
// J is cut into pieces of two rows by subtracting |beta| from both diagonal
// entries at every cut; pieces are merged pairwise.  A merge of two solved pieces is
// the rank-one update D + z z^T (D: both pieces' eigenvalues, z: the last row
// of the left and the first row of the right eigenvector matrix, times
// sqrt|beta|), whose eigenvalues are the roots of the secular equation
//     f(x) = 1 + sum_j z_j^2 / (d_j - x) = 0,
// one between neighbouring d_j: independent of one another, so they are found
// in parallel.  Only the first and last rows of the eigenvector matrices are
// carried, so a merge of size K costs O(K^2).  The parts, each as published:
//   * deflation of tiny z_j and of close d_j pairs (Dongarra & Sorensen 1987);
//   * the roots as offsets from the nearer pole, so that every d_j - x is
//     formed without cancellation, by rational interpolation with the two
//     neighbouring poles (Li 1993), inside a bracket;
//   * z recomputed from the computed roots by Loewner's formula, which keeps
//     the eigenvectors orthogonal to working precision whatever the spacing of
//     the roots (Gu & Eisenstat 1995).
//
// What bounds it: FP64 instructions.  One of a warp holds its scheduler's FP64
// unit for tens of cycles however few lanes are active, so the QR iteration of
// evc_tridiag.cuh -- a serial chain of about 0.85 k^2 rotations of some 45 of
// them -- took a count, which kept its scratch in shared memory, 2.3 ms at k = 40
// and 22 ms at k = 134 on one thread per column.
// Here the lanes of a block share the roots (P lanes per root, each summing
// every P-th term), and a root is first brought to FP32 accuracy in FP32 --
// its starting point only -- after which two FP64 evaluations suffice.
// Measured in the static call, whose QR has its scratch in global memory, 64
// columns (QR | this): k = 8 175 | 68 us, 40 3572 | 209 us, 134 36.2 | 1.0 ms, 256
// 137 | 2.1 ms; 4096 columns: k = 8 194 | 93 us, 16 690 | 279 us, 40 3.83 | 2.2 ms.
// Errors against LAPACK: the same 1e-15 (QR's too).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace evc {

constexpr double kDcEps = 2.220446049250313e-16;

// The lanes that work on one root: `P` consecutive lanes of a warp, of which
// this is lane `sub`.  sum() gives every lane the same bits.  A lane may do the
// work of WAY lanes instead: it keeps their partial sums apart and adds them in the
// order of the shuffles, so that the bits are those of WAY P lanes.
struct DcLanes {
    int sub, P;
    unsigned mask;
    template <typename R, int WAY>
    __host__ __device__ R sum(R (&v)[WAY]) const
    {
#pragma unroll
        for (int o = WAY >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < o; ++q) v[q] += v[q + o];
        R r = v[0];
#ifdef __CUDA_ARCH__
        for (int o = P >> 1; o > 0; o >>= 1) r += __shfl_xor_sync(mask, r, o);
#endif
        return r;
    }
    template <typename R, int WAY>
    __host__ __device__ R product(R (&v)[WAY]) const
    {
#pragma unroll
        for (int o = WAY >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < o; ++q) v[q] *= v[q + o];
        R r = v[0];
#ifdef __CUDA_ARCH__
        for (int o = P >> 1; o > 0; o >>= 1) r *= __shfl_xor_sync(mask, r, o);
#endif
        return r;
    }
};

// term(j, q) for this lane's j < K: j = sub + q P, q < WAY, and again WAY P further on.
template <int WAY, typename F>
__host__ __device__ inline void dc_each(int K, const DcLanes& g, F&& term)
{
    int j = g.sub;
    for (; j + (WAY - 1) * g.P < K; j += WAY * g.P)
#pragma unroll
        for (int q = 0; q < WAY; ++q) term(j + q * g.P, q);
#pragma unroll
    for (int q = 0; q < WAY - 1; ++q)
        if (j + q * g.P < K) term(j + q * g.P, q);
}

// 1/x to working precision: the hardware's approximation (20 bits) and two
// Newton steps, each of which squares the relative error: 2^-40, then the rounding
// of the last step, below 2 ulp.  x is a difference of distinct poles or of a pole and a root.
__host__ __device__ inline double dc_rcp(double x)
{
#ifdef __CUDA_ARCH__
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
#else
    return 1.0 / x;
#endif
}
__host__ __device__ inline float dc_rcp(float x)
{
#ifdef __CUDA_ARCH__
    return __fdividef(1.0f, x);
#else
    return 1.0f / x;
#endif
}
// A product that no compiler fuses with a sum (all sums of products here are fused,
// or not, in so many words: the variants of the solver have to agree bit by bit).
__host__ __device__ inline float dc_mul(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
__host__ __device__ inline double dc_rsqrt(double x)
{
#ifdef __CUDA_ARCH__
    return rsqrt(x);
#else
    return 1.0 / sqrt(x);
#endif
}

// psi, phi: the sums of z_j^2 / (d_j - x) over the poles left and right of the
// root; dpsi, dphi: their derivatives in x.
template <typename R>
struct DcSums {
    R psi, phi, dpsi, dphi;
};

// The step eta from x to the root of  c + s/(a_i - eta) + S/(a_j - eta), which
// matches f, psi' and phi' at x (a_i = d_i - x, a_j = d_j - x; Li's "middle
// way"), from A = a_i psi' and B = a_j phi'.  last: the root to the right of
// both poles.  In FP32: near the root no sum in it cancels, so eta keeps FP32's
// relative accuracy, and the next evaluation of f corrects the rest.
__host__ __device__ inline float dc_step(float ai, float aj, float A, float B, float f, bool last)
{
    const float c = f - A - B;
    const float a = fmaf(aj, f - A, ai * (f - B));
    const float b = ai * aj * f;
    const float disc = fmaf(a, a, -(4.0f * b * c));
    const float q = sqrtf(disc > 0.0f ? disc : 0.0f);
    float eta;
    if (last) eta = a >= 0.0f ? (a + q) / (2.0f * c) : 2.0f * b / (a - q);
    else eta = a <= 0.0f ? (a - q) / (2.0f * c) : 2.0f * b / (a + q);
    // f increases: the step must go against its sign (else Newton's step)
    if (!(f * eta < 0.0f)) eta = -f * ai * aj / fmaf(A, aj, B * ai);
    return eta;
}

// Poles and weights of one merge: K poles d (ascending, distinct) and z, and in
// FP32 for the starting points d = hi + lo and z2 = z^2.
struct DcPoles {
    const double *d, *z;
    const float *hi, *lo, *z2;
    int K;
};

template <int WAY>
__host__ __device__ inline DcSums<double> dc_sums(const DcPoles& p, int split, double org, double mu,
                                                  const DcLanes& g)
{
    // (the left sums are put aside at the first pole of a partial sum to the right: two
    // FP64 operations per term, not four)
    double psi[WAY] = {}, phi[WAY] = {}, dpsi[WAY] = {}, dphi[WAY] = {};
    dc_each<WAY>(p.K, g, [&](int j, int q) {
        const double zj = p.z[j];
        const double t = zj * dc_rcp((p.d[j] - org) - mu);
        if (j > split && j - WAY * g.P <= split) {
            psi[q] = phi[q];
            dpsi[q] = dphi[q];
            phi[q] = dphi[q] = 0.0;
        }
        phi[q] = fma(t, zj, phi[q]);
        dphi[q] = fma(t, t, dphi[q]);
    });
#pragma unroll
    for (int q = 0; q < WAY; ++q) {
        const int first = g.sub + q * g.P;               // no pole of this sum to the right:
        if (first + (p.K - 1 - first) / (WAY * g.P) * (WAY * g.P) <= split) {
            psi[q] = phi[q];
            dpsi[q] = dphi[q];
            phi[q] = dphi[q] = 0.0;
        }
    }
    return DcSums<double>{g.sum(psi), g.sum(phi), g.sum(dpsi), g.sum(dphi)};
}

template <int WAY>
__host__ __device__ inline DcSums<float> dc_sums(const DcPoles& p, int split, int o, float mu,
                                                 const DcLanes& g)
{
    const float hi = p.hi[o], lo = p.lo[o];
    float psi[WAY] = {}, phi[WAY] = {}, dpsi[WAY] = {}, dphi[WAY] = {};
    dc_each<WAY>(p.K, g, [&](int j, int q) {
        const float r = dc_rcp(((p.hi[j] - hi) + (p.lo[j] - lo)) - mu);
        const float v = dc_mul(p.z2[j], r), t = dc_mul(v, r);
        if (j <= split) {
            psi[q] += v;
            dpsi[q] += t;
        } else {
            phi[q] += v;
            dphi[q] += t;
        }
    });
    return DcSums<float>{g.sum(psi), g.sum(phi), g.sum(dpsi), g.sum(dphi)};
}

// 2^e and 2^-e for a normal x = m 2^e, 1 <= |m| < 2 (e within +-1022).
__host__ __device__ inline double dc_pow2(int e)
{
    const uint64_t b = (uint64_t)(e + 1023) << 52;
    double v;
    memcpy(&v, &b, 8);
    return v;
}
__host__ __device__ inline int dc_exp(double x)
{
    uint64_t b;
    memcpy(&b, &x, 8);
    const int e = (int)((b >> 52) & 2047) - 1023;
    return e < -1000 ? -1000 : e > 1000 ? 1000 : e;
}

// Root i of the secular equation, x_i = d[org] + mu: in (d_i, d_(i+1)), or for
// i = K - 1 in (d_i, d_i + sum z^2].
template <int WAY>
__host__ __device__ inline void dc_root(const DcPoles& p, int i, const DcLanes& g, int& org, double& mu)
{
    const int K = p.K;
    if (K == 1) {
        org = 0;
        mu = p.z[0] * p.z[0];
        return;
    }
    const bool last = i == K - 1;
    const int split = last ? K - 2 : i;              // poles d_split and d_(split+1) enter dc_step
    // ---- starting point in FP32
    const float gapf = (p.hi[split + 1] - p.hi[split]) + (p.lo[split + 1] - p.lo[split]);
    float lo32, hi32, m32;
    if (last) {
        org = K - 1;
        float zz[WAY] = {};
        dc_each<WAY>(K, g, [&](int j, int q) { zz[q] += p.z2[j]; });
        lo32 = 0.0f;
        hi32 = g.sum(zz);
        m32 = 0.5f * hi32;
    } else {
        const DcSums<float> s = dc_sums<WAY>(p, split, i, 0.5f * gapf, g);
        // f(middle) >= 0: the root lies in the left half
        org = 1.0f + s.psi + s.phi >= 0.0f ? i : i + 1;
        lo32 = org == i ? 0.0f : -gapf;
        hi32 = org == i ? gapf : 0.0f;
        m32 = 0.5f * (lo32 + hi32);
    }
    for (int it = 0; it < 20; ++it) {
        const DcSums<float> s = dc_sums<WAY>(p, split, org, m32, g);
        const float f = 1.0f + s.psi + s.phi;
        if (f < 0.0f) lo32 = m32;
        else hi32 = m32;
        const float ai = ((p.hi[split] - p.hi[org]) + (p.lo[split] - p.lo[org])) - m32;
        const float aj = ((p.hi[split + 1] - p.hi[org]) + (p.lo[split + 1] - p.lo[org])) - m32;
        const float eta = dc_step(ai, aj, ai * s.dpsi, aj * s.dphi, f, last);
        float nx = m32 + eta;
        // a root much nearer its pole than x is: the pole's term against the rest
        if (!(nx > lo32 && nx < hi32)) nx = p.z2[org] / (f + p.z2[org] / m32);
        if (!(nx > lo32 && nx < hi32)) nx = 0.5f * (lo32 + hi32);
        const bool done = fabsf(nx - m32) <= 1e-5f * fabsf(nx);
        m32 = nx;
        if (done) break;
    }
    // ---- FP64
    double lo, hi;
    const double dorg = p.d[org];
    if (last) {
        double zz[WAY] = {};
        dc_each<WAY>(K, g, [&](int j, int q) { zz[q] = fma(p.z[j], p.z[j], zz[q]); });
        lo = 0.0;
        hi = g.sum(zz) * (1.0 + 1e-12);
    } else {
        const double gap = p.d[i + 1] - p.d[i];
        lo = org == i ? 0.0 : -gap;
        hi = org == i ? gap : 0.0;
    }
    double x = (double)m32;
    if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
    const double di = p.d[split] - dorg, dj = p.d[split + 1] - dorg;
    for (int it = 0; it < 200; ++it) {
        const DcSums<double> s = dc_sums<WAY>(p, split, dorg, x, g);
        const double f = 1.0 + s.psi + s.phi;
        // f is known to the rounding of its terms
        if (fabs(f) <= 2.0 * kDcEps * (1.0 + fabs(s.psi) + fabs(s.phi))) break;
        if (f < 0.0) lo = x;
        else hi = x;
        // the step in units of x's power of two: FP32 has the range for it
        const double ai = di - x, aj = dj - x, unit = dc_pow2(dc_exp(x)), inv = dc_pow2(-dc_exp(x));
        double nx = x + unit * (double)dc_step((float)(ai * inv), (float)(aj * inv),
                                               (float)(ai * s.dpsi), (float)(aj * s.dphi), (float)f, last);
        if (!(nx > lo && nx < hi)) {
            const double z2 = p.z[org] * p.z[org];
            nx = z2 / (f + z2 / x);
            if (!(nx > lo && nx < hi)) nx = 0.5 * (lo + hi);
            if (!(nx > lo && nx < hi)) break;         // no number left between
            x = nx;
            continue;
        }
        // the next error is quadratic in this step
        const bool done = fabs(nx - x) <= 1e-9 * fabs(nx);
        x = nx;
        if (done) break;
    }
    mu = x;
}

// Loewner: the z_j (up to a common factor) for which the computed roots are
// exact: z_j^2 = (x_(K-1) - d_j) prod_(i<j) (x_i - d_j)/(d_i - d_j)
//                                prod_(j<=i<K-1) (x_i - d_j)/(d_(i+1) - d_j).
template <int WAY>
__host__ __device__ inline double dc_loewner(const DcPoles& p, const int* org, const double* mu, int j,
                                             const DcLanes& g)
{
    const double dj = p.d[j];
    double v[WAY];
#pragma unroll
    for (int q = 0; q < WAY; ++q) v[q] = 1.0;
    dc_each<WAY>(p.K, g, [&](int i, int q) {
        const double num = (p.d[org[i]] - dj) + mu[i];
        if (i == p.K - 1) v[q] *= num;
        else v[q] *= num * dc_rcp(p.d[i < j ? i : i + 1] - dj);
    });
    return copysign(sqrt(fabs(g.product(v))), p.z[j]);
}

// First and last components of the eigenvector of root i: of the normalised
// vector with entries zh_j / (d_j - x_i), against the rows F and L of the
// pieces' eigenvector matrices (lst: position of pole j in F and L).
template <int WAY>
__host__ __device__ inline void dc_vector(const DcPoles& p, const double* zh, const double* F,
                                          const double* L, const int* lst, int org, double mu,
                                          const DcLanes& g, bool want_last, double& first, double& lastc)
{
    const double dorg = p.d[org];
    double s[WAY] = {}, a[WAY] = {}, b[WAY] = {};
    dc_each<WAY>(p.K, g, [&](int j, int q) {
        const double u = zh[j] * dc_rcp((p.d[j] - dorg) - mu);
        s[q] = fma(u, u, s[q]);
        a[q] = fma(u, F[lst[j]], a[q]);
        if (want_last) b[q] = fma(u, L[lst[j]], b[q]);
    });
    const double inv = dc_rsqrt(g.sum(s));
    first = g.sum(a) * inv;
    lastc = g.sum(b) * inv;
}

// Close poles of one merge, in the order of its kept list: a pair whose
// rotation leaves an off-diagonal entry below tol is rotated so that the left
// one's z becomes zero, and that one is deflated.  Serial (rare).
__host__ __device__ inline bool dc_close(double dp, double dn, double zp, double zn, double tol)
{
    return fabs((dn - dp) * zp * zn) <= tol * (zp * zp + zn * zn);
}

__host__ __device__ inline void dc_deflate_close(double* D, double* Z, double* F, double* L,
                                                 const int* lst, unsigned char* gone, int K, double tol)
{
    int p = lst[0];
    for (int q = 1; q < K; ++q) {
        const int n = lst[q];
        if (dc_close(D[p], D[n], Z[p], Z[n], tol)) {
            const double tau = sqrt(Z[p] * Z[p] + Z[n] * Z[n]);
            const double c = Z[n] / tau, s = Z[p] / tau;
            const double fp = F[p], fn = F[n], lp = L[p], ln = L[n], dp = D[p], dn = D[n];
            Z[n] = tau;
            Z[p] = 0.0;
            F[n] = c * fn + s * fp;
            F[p] = c * fp - s * fn;
            L[n] = c * ln + s * lp;
            L[p] = c * lp - s * ln;
            D[p] = c * c * dp + s * s * dn;
            D[n] = s * s * dp + c * c * dn;
            gone[p] = 1;
        }
        p = n;
    }
}

// Rows t, t + 1 of the matrix as one solved piece: the rotation that
// diagonalises [p b; b q], eigenvalues ascending.
__host__ __device__ inline void dc_pair(double p, double b, double q, double* d, double* f, double* l)
{
    double c = 1.0, s = 0.0, t = 0.0;
    if (b != 0.0) {
        const double h = 0.5 * (q - p);
        // tan of the smaller angle: b / (|h| + sqrt(h^2 + b^2)), h's sign; entries
        // whose squares would vanish (b next to equal p and q) scaled up first
        const double sq = fma(b, b, h * h);
        if (sq < 1e-280) {
            const double hu = 0x1p+600 * h, bu = 0x1p+600 * b;
            t = bu / (fabs(hu) + sqrt(hu * hu + bu * bu));
        } else {
            t = b / (fabs(h) + sqrt(sq));
        }
        if (h < 0.0) t = -t;
        c = dc_rsqrt(1.0 + t * t);
        s = t * c;
    }
    const double x = p - t * b, y = q + t * b;     // vectors (c, -s) and (s, c)
    const int lo = x <= y ? 0 : 1;
    d[lo] = x;
    f[lo] = c;
    l[lo] = -s;
    d[1 - lo] = y;
    f[1 - lo] = s;
    l[1 - lo] = c;
}

// Shared-memory arrays of one matrix of order k: bytes of dc_solve's scratch.
__host__ __device__ inline size_t dc_smem(int k)
{
    // 11 double, 3 float, 3 int arrays and one byte array, rounded to 16 bytes
    return ((size_t)k * (11 * 8 + 3 * 4 + 3 * 4 + 1) + 15) & ~(size_t)15;
}

// Lanes per root and threads per block, by the order of the matrix alone (a
// column's bits must not depend on how many columns share the launch).  Up to
// 4 lanes: each repeats the scalar part of a step, so 16 lanes per root ran
// 1.6 times longer with 4096 columns of k = 16 (675 against 426 us) and no
// shorter with 64 (105 and 107 us).
__host__ __device__ inline int dc_lanes_per_root(int k, int nth)
{
    int P = 1;
    while (P < 4 && 2 * P * k <= nth) P <<= 1;
    return P;
}

struct DcWork {
    double *d, *f, *l;              // solved pieces: eigenvalues ascending, first and last rows
    double *D, *Z, *F, *L;          // a merge's poles in ascending order
    double *dc, *zc;                // ... those kept, contiguous
    double *mu, *zh;                // roots, Loewner's z
    float *hi, *lo, *z2;
    int *org, *lst, *cnt;           // root's pole, kept pole's row, kept poles (at a merge's first row)
    unsigned char* gone;            // deflated
};

__host__ __device__ inline DcWork dc_carve(void* base, int k)
{
    DcWork w;
    double* p = static_cast<double*>(base);
    double** dd[] = {&w.d, &w.f, &w.l, &w.D, &w.Z, &w.F, &w.L, &w.dc, &w.zc, &w.mu, &w.zh};
    for (double** q : dd) {
        *q = p;
        p += k;
    }
    float* fp = reinterpret_cast<float*>(p);
    w.hi = fp;
    w.lo = fp + k;
    w.z2 = fp + 2 * k;
    int* ip = reinterpret_cast<int*>(fp + 3 * k);
    w.org = ip;
    w.lst = ip + k;
    w.cnt = ip + 2 * k;
    w.gone = reinterpret_cast<unsigned char*>(ip + 3 * k);
    return w;
}

// Number of entries below v (strict) or up to v in the ascending list a[0..n).
__host__ __device__ inline int dc_below(const double* a, int n, double v, bool or_equal)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (a[m] < v || (or_equal && a[m] == v)) lo = m + 1;
        else hi = m;
    }
    return lo;
}

// The phases of one level, each run by every thread of the block (tid, nth)
// with a barrier after it.  e[t] couples rows t and t + 1; pieces have `half`
// rows (the last ones may be shorter), merge m covers rows [2 half m, 2 half
// (m + 1)) and is absent when its right piece is empty.
struct DcLevel {
    DcWork w;
    const double* e;
    int k, half, P;

    __host__ __device__ int beg(int g) const { return g / (2 * half) * (2 * half); }
    __host__ __device__ int mid(int g) const { return beg(g) + half; }
    __host__ __device__ int end(int g) const { const int b = beg(g) + 2 * half; return b < k ? b : k; }
    __host__ __device__ double tol(int g) const
    {
        const int b = beg(g);
        const double m = fmax(fmax(fabs(w.D[b]), fabs(w.D[end(g) - 1])), 2.0 * fabs(e[mid(g) - 1]));
        return 8.0 * kDcEps * m;
    }

    // poles in ascending order with their z and rows
    __host__ __device__ void sort(int tid, int nth) const
    {
        for (int g = tid; g < k; g += nth) {
            const int b = beg(g), m = mid(g), n = end(g);
            double dv = w.d[g];
            int at = g;
            double z = 0.0, f = w.f[g], l = w.l[g];
            if (m < n) {
                const double be = e[m - 1], rt = sqrt(fabs(be));
                if (g < m) {
                    at = g + dc_below(w.d + m, n - m, dv, false);
                    z = rt * l;
                    l = 0.0;
                } else {
                    at = b + (g - m) + dc_below(w.d + b, m - b, dv, true);
                    z = be < 0.0 ? -rt * f : rt * f;
                    f = 0.0;
                }
            }
            w.D[at] = dv;
            w.Z[at] = z;
            w.F[at] = f;
            w.L[at] = l;
        }
    }
    // tiny z
    __host__ __device__ void flag(int tid, int nth) const
    {
        for (int g = tid; g < k; g += nth) {
            const int m = mid(g);
            // (FP32 is enough to decide; what it flushes to zero is below 1e-38 of the norm)
            w.gone[g] = m >= end(g) ||
                        sqrtf(2.0f * fabsf((float)e[m - 1])) * fabsf((float)w.Z[g]) <= (float)tol(g);
        }
    }
    // the kept poles of a merge, contiguous from its first row
    __host__ __device__ void keep(int tid, int nth) const
    {
        for (int g = tid; g < k; g += nth) {
            const int b = beg(g);
            int at = b;
            for (int j = b; j < g; ++j) at += !w.gone[j];
            if (g == end(g) - 1) w.cnt[b] = at - b + !w.gone[g];
            if (w.gone[g]) continue;
            w.lst[at] = g;
            w.dc[at] = w.D[g];
            w.zc[at] = w.Z[g];
            const float h = (float)w.D[g];
            w.hi[at] = h;
            w.lo[at] = (float)(w.D[g] - (double)h);
            w.z2[at] = (float)(w.Z[g] * w.Z[g]);
        }
    }
    __host__ __device__ int kept(int g) const { return w.cnt[beg(g)]; }
    // whether row g is a kept pole that is too close to the next kept one
    __host__ __device__ bool close(int g) const
    {
        const int b = beg(g), K = kept(g);
        const int q = g - b;                         // as a position in the kept list
        return q + 1 < K && dc_close(w.dc[g], w.dc[g + 1], w.zc[g], w.zc[g + 1], tol(g));
    }
    __host__ __device__ void deflate_close(int b) const
    {
        const int K = kept(b);
        if (K > 1) dc_deflate_close(w.D, w.Z, w.F, w.L, w.lst + b, w.gone, K, tol(b));
    }
    __host__ __device__ DcPoles poles(int g) const
    {
        const int b = beg(g);
        return DcPoles{w.dc + b, w.zc + b, w.hi + b, w.lo + b, w.z2 + b, kept(g)};
    }
    template <int WAY>
    __host__ __device__ void roots(int g, const DcLanes& ln) const
    {
        const int b = beg(g), i = g - b;
        const DcPoles p = poles(g);
        if (i >= p.K) return;
        int org;
        double mu;
        dc_root<WAY>(p, i, ln, org, mu);
        if (ln.sub == 0) {
            w.org[g] = org;
            w.mu[g] = mu;
        }
    }
    template <int WAY>
    __host__ __device__ void loewner(int g, const DcLanes& ln) const
    {
        const int b = beg(g), i = g - b;
        const DcPoles p = poles(g);
        if (i >= p.K) return;
        const double v = dc_loewner<WAY>(p, w.org + b, w.mu + b, i, ln);
        if (ln.sub == 0) w.zh[g] = v;
    }
    // rows of the new eigenvectors, into d, f, l: the roots first, then the
    // deflated poles, in no order yet
    template <int WAY>
    __host__ __device__ void vectors(int g, const DcLanes& ln) const
    {
        const int b = beg(g), i = g - b;
        const DcPoles p = poles(g);
        if (i < p.K) {
            double a, c;
            const int org = w.org[g];
            const double mu = w.mu[g];
            dc_vector<WAY>(p, w.zh + b, w.F, w.L, w.lst + b, org, mu, ln, 2 * half < k, a, c);
            if (ln.sub == 0) {
                w.d[g] = p.d[org] + mu;
                w.f[g] = a;
                w.l[g] = c;
            }
        }
        if (ln.sub == 0 && w.gone[g]) {
            int at = b + p.K;
            for (int j = b; j < g; ++j) at += w.gone[j];
            w.d[at] = w.D[g];
            w.f[at] = w.F[g];
            w.l[at] = w.L[g];
        }
    }
    // ascending order again, into D, F and L
    __host__ __device__ void order(int tid, int nth) const
    {
        for (int g = tid; g < k; g += nth) {
            const int b = beg(g), n = end(g);
            const double v = w.d[g];
            int at = g;
            if (kept(g) < n - b) {
                at = b;
                for (int j = b; j < n; ++j) at += w.d[j] < v || (w.d[j] == v && j < g);
            }
            w.D[at] = v;
            w.F[at] = w.f[g];
            w.L[at] = w.l[g];
        }
    }
    __host__ __device__ void swap()
    {
        double* t = w.d;
        w.d = w.D;
        w.D = t;
        t = w.f;
        w.f = w.F;
        w.F = t;
        t = w.l;
        w.l = w.L;
        w.L = t;
    }
};

// Threads that work on a matrix of order k.
__host__ __device__ inline int dc_threads(int k) { return k <= 8 ? 32 : k <= 16 ? 64 : k <= 32 ? 128 : k <= 128 ? 256 : 512; }

#ifdef __CUDACC__
// The whole block solves one matrix of order k >= 1: w.d its diagonal, e[0..k-1)
// its off-diagonal, both in shared memory and overwritten.  On return w.d holds
// the eigenvalues times 2^-ex, ascending, and w.f the first components of the
// eigenvectors; false (for every thread) when an entry is not finite.  Every
// thread of the block calls it; blockDim.x >= dc_threads(k), and the result
// depends on k and the entries only.
__device__ inline bool dc_solve(DcWork& w, double* e, int k, int& ex)
{
    const int tid = threadIdx.x, nth = dc_threads(k);
    __shared__ int s_ex;
    if (tid == 0) s_ex = -100000;
    __syncthreads();
    int mx = -100000, bad = 0;
    for (int t = tid; t < k; t += blockDim.x) {
        const double a = fabs(w.d[t]), b = t + 1 < k ? fabs(e[t]) : 0.0;
        bad |= !isfinite(a) || !isfinite(b);
        const double m = fmax(a, b);
        if (m > 0.0 && isfinite(m)) mx = max(mx, ilogb(m) + 1);
    }
    if (mx > -100000) atomicMax(&s_ex, mx);
    if (__syncthreads_or(bad)) return false;
    ex = s_ex > -100000 ? s_ex : 0;
    // scaled to a largest entry in [1/2, 1) (a power of two: exact), then cut
    for (int t = tid; t < k; t += blockDim.x) {
        w.d[t] = scalbn(w.d[t], -ex);
        if (t + 1 < k) e[t] = scalbn(e[t], -ex);
        w.f[t] = w.l[t] = 1.0;
    }
    __syncthreads();
    for (int t = 2 * tid; t < k; t += 2 * blockDim.x) {
        const double a = t > 0 ? fabs(e[t - 1]) : 0.0, b = t + 2 < k ? fabs(e[t + 1]) : 0.0;
        if (t + 1 < k) dc_pair(w.d[t] - a, e[t], w.d[t + 1] - b, w.d + t, w.f + t, w.l + t);
        else w.d[t] -= a;
    }
    __syncthreads();
    const int P = dc_lanes_per_root(k, nth);
    const int grp = tid / P, ngrp = nth / P;
    const DcLanes ln{tid % P, P, ((1u << P) - 1u) << ((tid & 31) & ~(P - 1))};
    const bool on = tid < nth;
    for (int half = 2; half < k; half *= 2) {
        DcLevel L{w, e, k, half, P};
        if (on) L.sort(tid, nth);
        __syncthreads();
        if (on) L.flag(tid, nth);
        __syncthreads();
        if (on) L.keep(tid, nth);
        __syncthreads();
        int any = 0;
        if (on)
            for (int g = tid; g < k; g += nth) any |= L.close(g);
        if (__syncthreads_or(any)) {
            if (on)
                for (int g = tid; g < k; g += nth)
                    if (L.beg(g) == g) L.deflate_close(g);
            __syncthreads();
            if (on) L.keep(tid, nth);
            __syncthreads();
        }
        if (on)
            for (int g = grp; g < k; g += ngrp) L.roots<1>(g, ln);
        __syncthreads();
        if (on)
            for (int g = grp; g < k; g += ngrp) L.loewner<1>(g, ln);
        __syncthreads();
        if (on)
            for (int g = grp; g < k; g += ngrp) L.vectors<1>(g, ln);
        __syncthreads();
        if (on) L.order(tid, nth);
        __syncthreads();
        L.swap();
        w = L.w;
    }
    return true;
}

// The same for many matrices of up to 32 rows, several in a warp (lane `base` + t: row
// t < kmax of a matrix of k <= kmax rows, kmax the same in all lanes; k = 0: none): one
// lane per root, which keeps apart the partial sums of the four lanes that it has
// above, so that the bits are the same.  All 32 lanes of the warp call it.
// For a block per matrix the scalar part of a step, which every lane repeats, and the
// rows that fill no warp take most of the FP64 units' time once there are matrices
// enough.  us, block per matrix | packed (64 registers, 32 warps per SM): 4096 matrices
// k = 4 72 | 33, 8 137 | 93, 16 410 | 279, 32 1177 | 818; 16384 k = 5 509 | 157, 8 528 | 231,
// 12 1190 | 791, 16 1449 | 858; 1024 k = 8 72 | 70, 16 132 | 125, 20 201 | 247.  (One thread
// per matrix, evc_tridiag.cuh, with 16384: 82, 195, 406 and 699, other bits.)
__device__ inline bool dc_solve_packed(DcWork& w, double* e, int k, int kmax, int base, int tid, int& ex)
{
    const unsigned group = (kmax == 32 ? 0xffffffffu : (1u << kmax) - 1u) << base;
    int mx = -100000, bad = 0;
    if (tid < k) {
        const double a = fabs(w.d[tid]), b = tid + 1 < k ? fabs(e[tid]) : 0.0;
        bad = !isfinite(a) || !isfinite(b);
        const double m = fmax(a, b);
        if (m > 0.0 && isfinite(m)) mx = ilogb(m) + 1;
    }
    ex = -100000;
    for (int t = 0; t < kmax; ++t) ex = max(ex, __shfl_sync(0xffffffffu, mx, min(base + t, 31)));
    if (ex == -100000) ex = 0;
    if (__ballot_sync(0xffffffffu, bad) & group) k = 0;     // (its lanes stay for the barriers)
    const bool ok = k > 0;
    if (tid < k) {
        w.d[tid] = scalbn(w.d[tid], -ex);
        if (tid + 1 < k) e[tid] = scalbn(e[tid], -ex);
        w.f[tid] = w.l[tid] = 1.0;
    }
    __syncwarp();
    if (2 * tid < k) {
        const int t = 2 * tid;
        const double a = t > 0 ? fabs(e[t - 1]) : 0.0, b = t + 2 < k ? fabs(e[t + 1]) : 0.0;
        if (t + 1 < k) dc_pair(w.d[t] - a, e[t], w.d[t + 1] - b, w.d + t, w.f + t, w.l + t);
        else w.d[t] -= a;
    }
    __syncwarp();
    const DcLanes ln{0, 1, 0};
    for (int half = 2; half < kmax; half *= 2) {
        DcLevel lv{w, e, k, half, 1};
        const bool act = half < k && tid < k;
        if (act) lv.sort(tid, kmax);
        __syncwarp();
        if (act) lv.flag(tid, kmax);
        __syncwarp();
        if (act) lv.keep(tid, kmax);
        __syncwarp();
        const bool close = __ballot_sync(0xffffffffu, act && lv.close(tid)) & group;
        if (close && act && lv.beg(tid) == tid) lv.deflate_close(tid);
        __syncwarp();
        if (close && act) lv.keep(tid, kmax);
        __syncwarp();
        if (act) lv.roots<4>(tid, ln);
        __syncwarp();
        if (act) lv.loewner<4>(tid, ln);
        __syncwarp();
        if (act) lv.vectors<4>(tid, ln);
        __syncwarp();
        if (act) lv.order(tid, kmax);
        __syncwarp();
        if (half < k) {
            lv.swap();
            w = lv.w;
        }
    }
    return ok;
}

// Sum of the squared first components over the eigenvalues below sigma, by the
// lanes of one warp (a fixed order for a given k).
__device__ inline double dc_weight_below(const DcWork& w, int k, int ex, double sigma)
{
    const double s = scalbn(sigma, -ex);
    double q = 0.0;
    for (int t = threadIdx.x & 31; t < k; t += 32)
        if (w.d[t] < s) q += w.f[t] * w.f[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    return q;
}
// The same for packed matrices, in lane tid = 0: the additions of that tree whose
// terms are not zero by their place.
__device__ inline double dc_weight_below_packed(const DcWork& w, int k, int ex, int base, int tid, double sigma)
{
    double q = tid < k && w.d[tid] < scalbn(sigma, -ex) ? w.f[tid] * w.f[tid] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double v = __shfl_sync(0xffffffffu, q, min(base + tid + o, 31));
        if (tid < o && tid + o < k) q += v;
    }
    return q;
}

// Packed matrices: threads per block, matrices per block, and bytes of shared memory of
// a matrix of up to k rows.
constexpr int kPackedThreads = 128, kPackedBlocks = 8;   // (blocks per SM: 64 registers)
__host__ __device__ inline bool dc_packed_pays(int k, int matrices) { return k <= 16 ? matrices >= 1024 : k <= 32 && matrices >= 4096; }
__host__ __device__ inline int dc_packed_matrices(int k) { return kPackedThreads / 32 * (32 / k); }
__host__ __device__ inline size_t dc_packed_bytes(int k) { return dc_smem(k) + (size_t)((k + 1) & ~1) * sizeof(double); }
// This lane's matrix among the block's (-1: none) and its place in it.
struct DcPlace {
    int at, base, tid;
};
__device__ inline DcPlace dc_packed_place(int k)
{
    const int lane = threadIdx.x & 31, per = 32 / k, in = lane / k;
    // (the lanes left over read the last matrix's lanes in the shuffles)
    return in < per ? DcPlace{(int)(threadIdx.x >> 5) * per + in, in * k, lane - in * k} : DcPlace{-1, 0, 32};
}
#endif

}  // namespace evc
