// Pippenger multi-scalar multiplication over BLS12-377 G1 (Sec. II-C of the
// paper: windows, bucket accumulation, bucket aggregation, group aggregation),
// laid out for one GB300.
//
// Stages:
//  1. prepare     standard affine -> Montgomery affine (96 B per point, AoS, so a
//                 random gather of one point reads three full 32 B sectors)
//  2. digits      c-bit window digits per scalar (signed or unsigned);
//                 |digit| and its sign, window-major
//  3. sort        point indices in bucket order within each window: a counting sort
//                 over (window, key) bins (count, scan, scatter), or a stable LSD
//                 radix sort with 8-bit digits per pass
//  4. accumulate  every bucket's run of points is cut into pieces of bounded length;
//                 the pieces, longest first, are summed with mixed PADDs, one thread
//                 each, so the lanes of a warp add equally many points
//  5. merge       the pieces of buckets that needed more than one are added up
//  6. reduce      per window sum_b b * B_b: segments of L buckets by running sums
//                 in-thread, then sum_g g * Y_g split by the bits of g into
//                 independent sums, recombined by Horner
//  7. combine     sum_j 2^(c j) S_j by Horner over windows, one inversion,
//                 affine standard form
//
// Everything runs on the caller's stream, one launch per stage over all windows.
//
// Two curve models run the same pipeline (a template parameter of every point
// kernel): short Weierstrass XYZZ (default; any points on the curve) and the
// paper's twisted Edwards model in extended coordinates (MSM377_EDWARDS; 7M
// mixed additions, points of the order-r subgroup). MSM377_GLV splits every
// scalar k = k1 + lambda k2 (lambda = x0^2 - 1, 127-bit halves) and runs the
// pipeline over the 2n points P_i, phi(P_i) = (beta x_i, y_i) with half the
// windows (subgroup points); stored rows 2i and 2i + 1 are P_i and phi(P_i).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "ec.cuh"
#include "ed.cuh"
#include "wred.cuh"

namespace {

using ec::affine;
using ec::xyzz;
using fq::fe;

constexpr uint32_t kNone = 0xffffffffu;
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;  // 2048
constexpr int kXyzzVec = 12;                // XYZZ in memory: 4 x 12 packed words = 12 uint4
constexpr size_t kXyzzBytes = kXyzzVec * 16;

// ---------------------------------------------------------------- memory I/O

__device__ __forceinline__ void load_affine(affine& Q, const uint4* __restrict__ pts, uint32_t idx) {
    const uint4* p = pts + 6 * (size_t)idx;
    uint4 a = __ldg(p + 0), b = __ldg(p + 1), c = __ldg(p + 2);
    uint4 d = __ldg(p + 3), e = __ldg(p + 4), f = __ldg(p + 5);
    Q.x.v[0] = a.x; Q.x.v[1] = a.y; Q.x.v[2] = a.z; Q.x.v[3] = a.w;
    Q.x.v[4] = b.x; Q.x.v[5] = b.y; Q.x.v[6] = b.z; Q.x.v[7] = b.w;
    Q.x.v[8] = c.x; Q.x.v[9] = c.y; Q.x.v[10] = c.z; Q.x.v[11] = c.w;
    Q.y.v[0] = d.x; Q.y.v[1] = d.y; Q.y.v[2] = d.z; Q.y.v[3] = d.w;
    Q.y.v[4] = e.x; Q.y.v[5] = e.y; Q.y.v[6] = e.z; Q.y.v[7] = e.w;
    Q.y.v[8] = f.x; Q.y.v[9] = f.y; Q.y.v[10] = f.z; Q.y.v[11] = f.w;
}

__device__ __forceinline__ void load_fe(fe& a, const uint4* p) {
    uint4 u0 = p[0], u1 = p[1], u2 = p[2];
    a.v[0] = u0.x; a.v[1] = u0.y; a.v[2] = u0.z; a.v[3] = u0.w;
    a.v[4] = u1.x; a.v[5] = u1.y; a.v[6] = u1.z; a.v[7] = u1.w;
    a.v[8] = u2.x; a.v[9] = u2.y; a.v[10] = u2.z; a.v[11] = u2.w;
}

__device__ __forceinline__ void store_fe(uint4* p, const fe& a) {
    p[0] = make_uint4(a.v[0], a.v[1], a.v[2], a.v[3]);
    p[1] = make_uint4(a.v[4], a.v[5], a.v[6], a.v[7]);
    p[2] = make_uint4(a.v[8], a.v[9], a.v[10], a.v[11]);
}

// XYZZ point in memory: 12 uint4 (X, Y, ZZ, ZZZ), each coordinate in [0, 2p).
__device__ __forceinline__ void load_xyzz(xyzz& P, const uint4* p) {
    load_fe(P.X, p);
    load_fe(P.Y, p + 3);
    load_fe(P.ZZ, p + 6);
    load_fe(P.ZZZ, p + 9);
}

__device__ __forceinline__ void store_xyzz(uint4* p, const xyzz& P) {
    store_fe(p, P.X);
    store_fe(p + 3, P.Y);
    store_fe(p + 6, P.ZZ);
    store_fe(p + 9, P.ZZZ);
}

// Second operand of ec::add_q() read from memory coordinate by coordinate.
struct MemQ {
    const uint4* p;
    __device__ __forceinline__ void X(fe& r) const { load_fe(r, p); }
    __device__ __forceinline__ void Y(fe& r) const { load_fe(r, p + 3); }
    __device__ __forceinline__ void ZZ(fe& r) const { load_fe(r, p + 6); }
    __device__ __forceinline__ void ZZZ(fe& r) const { load_fe(r, p + 9); }
    __device__ __forceinline__ void all(xyzz& r) const { load_xyzz(r, p); }
};

// Second operand of ed::add_q() read from memory: (X, Y, Z, T) as 12 uint4.
struct MemQE {
    const uint4* p;
    __device__ __forceinline__ void X(fe& r) const { load_fe(r, p); }
    __device__ __forceinline__ void Y(fe& r) const { load_fe(r, p + 3); }
    __device__ __forceinline__ void Z(fe& r) const { load_fe(r, p + 6); }
    __device__ __forceinline__ void T(fe& r) const { load_fe(r, p + 9); }
};

// ---------------------------------------------------------------- curve models
//
// What the pipeline needs from a curve model: the stored form of an input point
// (kStored uint4 per point), a mixed addition of a gathered stored point, a full
// addition from memory or registers, a doubling, and the affine Weierstrass
// result. Accumulators of both models are four 12-word coordinates, 12 uint4 in
// memory. A bucket that received no point is all-zero words in memory: XYZZ
// reads that as its identity (ZZ = 0); the Edwards loader skips it.

struct ModelXyzz {
    using acc = xyzz;
    static constexpr int kAccBlocks = 3;  // accumulation blocks of 128 per SM (<= 168 registers)
    static constexpr int kStored = 6;  // affine (x, y)
    static __device__ __forceinline__ void set_inf(acc& P) { ec::set_inf(P); }
    static __device__ __forceinline__ void load(acc& P, const uint4* p) { load_xyzz(P, p); }
    static __device__ __forceinline__ void store(uint4* p, const acc& P) { store_xyzz(p, P); }
    static __device__ __forceinline__ bool first_at(acc& P, const uint4* pts, uint32_t idx, bool negate) {
        affine Q;
        load_affine(Q, pts, idx);
        if (negate) ec::neg(Q);
        ec::from_affine(P, Q);
        return ec::is_inf(Q);
    }
    static __device__ __forceinline__ void madd_at(acc& P, bool& inf, const uint4* pts, uint32_t idx, bool negate) {
        affine Q;
        load_affine(Q, pts, idx);
        if (negate) ec::neg(Q);
        ec::madd(P, inf, Q);
    }
    static __device__ __forceinline__ bool empty(const uint4*) { return false; }  // ZZ = 0 is the identity
    static __device__ __forceinline__ void add_mem(acc& P, const uint4* q) { ec::add_q(P, MemQ{q}); }
    static __device__ __forceinline__ void add(acc& P, const acc& Q) { ec::add(P, Q); }
    static __device__ __forceinline__ void add4_mem(acc& P, const uint4* q, fe* sh, int l) {
        ec::add4(P, MemQ{q}, sh, l, true);
    }
    static __device__ __forceinline__ void exchange(acc& Q, const acc& P);   // the neighbour lane's point
    using chain = wred::Weierstrass;  // four-warp group operations (wred.cuh)
};

struct ModelEdwards {
    using acc = ed::ext;
    static constexpr int kAccBlocks = 4;  // accumulation blocks of 128 per SM (<= 128 registers)
    static constexpr int kStored = 9;  // (x, y, u = k x y), the paper's (X, Y, U) with Z = 1
    static __device__ __forceinline__ void set_inf(acc& P) { ed::set_inf(P); }
    static __device__ __forceinline__ void load(acc& P, const uint4* p) {
        load_fe(P.X, p);
        load_fe(P.Y, p + 3);
        load_fe(P.Z, p + 6);
        load_fe(P.T, p + 9);
    }
    static __device__ __forceinline__ void store(uint4* p, const acc& P) {
        store_fe(p, P.X);
        store_fe(p + 3, P.Y);
        store_fe(p + 6, P.Z);
        store_fe(p + 9, P.T);
    }
    static __device__ __forceinline__ void load_stored(ed::stored& Q, const uint4* pts, uint32_t idx, bool negate) {
        const uint4* q = pts + (size_t)kStored * idx;
        load_fe(Q.x, q);
        load_fe(Q.y, q + 3);
        load_fe(Q.u, q + 6);
        if (negate) ed::neg(Q);
    }
    // acc <- the first point; the flag says acc is the identity (never, here)
    static __device__ __forceinline__ bool first_at(acc& P, const uint4* pts, uint32_t idx, bool negate) {
        ed::stored Q;
        load_stored(Q, pts, idx, negate);
        ed::from_stored(P, Q);
        return false;
    }
    static __device__ __forceinline__ void madd_at(acc& P, bool&, const uint4* pts, uint32_t idx, bool negate) {
        ed::stored Q;
        load_stored(Q, pts, idx, negate);
        ed::madd(P, Q);
    }
    static __device__ __forceinline__ bool empty(const uint4* q) {
        fe z;
        load_fe(z, q + 6);
        return fq::is_zero_raw(z);
    }
    static __device__ __forceinline__ void add_mem(acc& P, const uint4* q) {
        if (!empty(q)) ed::add_q(P, MemQE{q});
    }
    static __device__ __forceinline__ void add(acc& P, const acc& Q) { ed::add(P, Q); }
    static __device__ __forceinline__ void add4_mem(acc& P, const uint4* q, fe* sh, int l) {
        ed::add4(P, MemQE{q}, sh, l, true);
    }
    static __device__ __forceinline__ void exchange(acc& Q, const acc& P);
    using chain = wred::Edwards;
};

// ---------------------------------------------------------------- stage 1

// beta, a primitive cube root of unity in Fq with (beta x, y) = lambda (x, y) on
// the order-r subgroup (Montgomery form).
__device__ __constant__ static const uint32_t kBeta[fq::N] = {
    0xa5847973u, 0xdacd106du, 0xbac2a79au, 0xd8fe2454u, 0xfd832edcu, 0x1ada4fd6u,
    0x9d150908u, 0xfb986844u, 0xea32285eu, 0xd63eb8aeu, 0x6f873fd0u, 0x0167d6a3u};

// Stored point i of np in Montgomery form: input point i when np = n; with GLV
// (np = 2n) rows 2j and 2j + 1 are P_j and phi(P_j) = (beta x_j, y_j), so any
// contiguous range of input points is a contiguous range of stored rows. The
// affine identity (0, 0) stays (0, 0).
__device__ __forceinline__ void glv_source(fe& x, fe& y, const uint4* __restrict__ in, size_t i, size_t n,
                                           size_t np) {
    const bool split = np != n;
    const size_t src = split ? i >> 1 : i;
    load_fe(x, in + 6 * src);
    load_fe(y, in + 6 * src + 3);
    fq::to_mont(x, x);
    fq::to_mont(y, y);
    if (split && (i & 1)) {
        fe b;
        ed::load_const(b, kBeta);
        fq::mul(x, x, b);
        fq::canon(x, x);
    }
}

// Stored rows [lo, hi) of np (the whole set: lo = 0, hi = np).
__global__ void k_prepare(const uint4* __restrict__ in, uint4* __restrict__ out, size_t n, size_t np, size_t lo,
                          size_t hi) {
    size_t i = lo + blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= hi) return;
    fe x, y;
    glv_source(x, y, in, i, n, np);
    store_fe(out + 6 * i, x);
    store_fe(out + 6 * i + 3, y);
}

// Weierstrass -> Edwards stored form. For (x_w, y_w), with a = x_w + 1:
//   D = y_w (a + s),  x = c1 a (a + s) / D,  y = (a - s) y_w / D,  u = k x y.
// The affine identity, and points outside the map's domain (D = 0: order 2 or 4,
// never in the subgroup), become the Edwards identity (0, 1, 0).
//
// ed_affine_chunk (used by the fixed-base precomputation) takes kEdChunk points
// per lane in registers: one inversion per warp (Montgomery's trick twice: each
// thread multiplies the D of its kEdChunk points, a warp scan multiplies the
// threads' products, lane 0 inverts the warp's total, and prefix and suffix
// products hand every thread the inverse of its own product, from which it walks
// back through its chunk). k_prepare_ed, below, is the same map arranged for the
// preparation of whole sets.
constexpr int kEdChunk = 8;
// The GLV pair path of ed_affine_chunk needs every lane's first row and row count
// even (pairs P, phi(P) never straddle two lanes).
static_assert(kEdChunk % 2 == 0, "kEdChunk must be even");

__device__ __forceinline__ fe shfl_fe_up(const fe& a, int off) {
    fe r;
#pragma unroll
    for (int k = 0; k < fq::N; ++k) r.v[k] = __shfl_up_sync(0xffffffffu, a.v[k], off);
    return r;
}

__device__ __forceinline__ fe shfl_fe_down(const fe& a, int off) {
    fe r;
#pragma unroll
    for (int k = 0; k < fq::N; ++k) r.v[k] = __shfl_down_sync(0xffffffffu, a.v[k], off);
    return r;
}

__device__ __forceinline__ fe shfl_fe(const fe& a, int src) {
    fe r;
#pragma unroll
    for (int k = 0; k < fq::N; ++k) r.v[k] = __shfl_sync(0xffffffffu, a.v[k], src);
    return r;
}

// The inverse of every lane's acc (nonzero on every lane) with one field inversion
// for the warp: prefix products P_l = acc_0 ... acc_l and suffix products
// S_l = acc_{l+1} ... acc_31 over the lanes give acc_l^-1 = total^-1 P_{l-1} S_l.
// Every lane of the warp must call it. This form, a binary GCD on lane 0 and the two scans
// one after the other, is the faster one in the fixed-base precomputation, whose doublings
// keep the multiply pipe busy meanwhile (20000 points, c = 13: 9.5 ms, with the form below
// 10.3).
__device__ __forceinline__ fe warp_lane_inverse(const fe& acc) {
    const int lane = threadIdx.x & 31;
    fe one;
    fq::set_one(one);
    fe pre = acc, y;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {  // P_l
        y = shfl_fe_up(pre, off);
        if (lane >= off) fq::mul(pre, pre, y);
    }
    fe sacc = acc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {  // acc_l ... acc_31
        y = shfl_fe_down(sacc, off);
        if (lane + off < 32) fq::mul(sacc, sacc, y);
    }
    fe suf = shfl_fe_down(sacc, 1);           // S_l
    if (lane == 31) suf = one;
    const fe total = shfl_fe(pre, 31);
    fe tinv = one;
    if (lane == 0) ec::inv(tinv, total);
    tinv = shfl_fe(tinv, 0);
    fe before = shfl_fe_up(pre, 1);           // P_{l-1}
    if (lane == 0) before = one;
    fe inv;
    fq::mul(inv, tinv, before);
    fq::mul(inv, inv, suf);
    return inv;
}

// The same with the inversion on all lanes (wred::inverse) and the scans paired, for the
// preparation, which waits for it: 300007 GLV pairs 389 -> 309 us, 2^20 930 -> 857. mem:
// wred::kInverseWords words of shared memory of this warp's own.
__device__ __forceinline__ fe warp_lane_inverse_wide(const fe& acc, uint32_t* mem) {
    const int lane = threadIdx.x & 31;
    fe one;
    fq::set_one(one);
    fe pre = acc, sacc = acc, y;              // P_l; acc_l ... acc_31
#pragma unroll 1
    for (int off = 1; off < 32; off <<= 1) {
        y = shfl_fe_up(pre, off);
        fe z = shfl_fe_down(sacc, off);
        fq::mul2(y, pre, y, z, sacc, z);
        if (lane >= off) pre = y;
        if (lane + off < 32) sacc = z;
    }
    fe suf = shfl_fe_down(sacc, 1);           // S_l
    if (lane == 31) suf = one;
    const fe tinv = wred::inverse_fe(pre, 31, mem);
    fe before = shfl_fe_up(pre, 1);           // P_{l-1}
    if (lane == 0) before = one;
    fe inv;
    fq::mul(inv, tinv, before);
    fq::mul(inv, inv, suf);
    return inv;
}

// Replaces den[j] (j < m, where ok[j]) by its inverse, with one inversion for
// the whole warp: each lane multiplies its chunk, warp_lane_inverse hands it the
// inverse of that product, from which it walks back through its chunk. Every lane
// of the warp must call it (m may be 0; lanes carry 1 then).
template <int K>
__device__ __forceinline__ void warp_batch_inverse(fe (&den)[K], const bool (&ok)[K], int m) {
    fe prefix[K];
    fe acc;
    fq::set_one(acc);
    for (int j = 0; j < m; ++j) {
        prefix[j] = acc;                   // product of the valid den[0..j-1]
        if (ok[j]) fq::mul(acc, acc, den[j]);
    }
    fe inv = warp_lane_inverse(acc);
    for (int j = m - 1; j >= 0; --j) {
        if (!ok[j]) continue;
        fe dj;
        fq::mul(dj, inv, prefix[j]);
        fq::mul(inv, inv, den[j]);
        den[j] = dj;
    }
}

__device__ __forceinline__ void store_ed_identity(uint4* o) {
    fe z, one;
    fq::set_zero(z);
    fq::set_one(one);
    fq::canon(one, one);
    store_fe(o, z);
    store_fe(o + 3, one);
    store_fe(o + 6, z);
}

// Edwards affine (x, y) of the chunk's stored points i0 .. i0 + m - 1 (from the
// standard-form input, GLV rows included); ok[j] is false for the affine identity
// and points outside the map's domain, whose (x, y) is then left unset. Every lane
// of the warp must call it (one inversion per warp).
// pairs: GLV rows taken as (P, phi(P)) pairs. The caller decides it for the whole
// launch (every lane must reach the same warp_batch_inverse): a GLV row range with
// an even start and end, so every lane's i0 and m are even.
__device__ __forceinline__ void ed_affine_chunk(const uint4* __restrict__ in, size_t n, size_t np, size_t i0, int m,
                                                bool pairs, fe (&xe)[kEdChunk], fe (&ye)[kEdChunk],
                                                bool (&ok)[kEdChunk]) {
    fe one, sp;
    fq::set_one(one);
    ed::load_const(sp, ed::kS);
    if (pairs) {
        // GLV rows in pairs (P, phi(P)) = ((x, y), (beta x, y)): the pair shares y, so
        // it inverts y, a + s and a' + s (a = x + 1, a' = beta x + 1) instead of the
        // two products y (a + s), y (a' + s); x_e = c1 a / y, y_e = (a - s) / (a + s).
        constexpr int kPairs = kEdChunk / 2;
        fe xs[kEdChunk], inv[3 * kPairs];
        bool okv[3 * kPairs];
        fe y[kPairs];
        for (int q = 0; q < m / 2; ++q) {
            fe x0;
            glv_source(x0, y[q], in, i0 + 2 * q, n, np);
            const bool id = fq::is_zero_raw(x0) && fq::is_zero_raw(y[q]);
            fe b;
            ed::load_const(b, kBeta);
            fq::mul(xs[2 * q + 1], x0, b);
            fq::canon(xs[2 * q + 1], xs[2 * q + 1]);
            xs[2 * q] = x0;
            inv[3 * q] = y[q];
            fq::add(inv[3 * q + 1], xs[2 * q], one);
            fq::add(inv[3 * q + 1], inv[3 * q + 1], sp);
            fq::add(inv[3 * q + 2], xs[2 * q + 1], one);
            fq::add(inv[3 * q + 2], inv[3 * q + 2], sp);
            okv[3 * q] = !id && !fq::is_zero(inv[3 * q]);
            okv[3 * q + 1] = !id && !fq::is_zero(inv[3 * q + 1]);
            okv[3 * q + 2] = !id && !fq::is_zero(inv[3 * q + 2]);
        }
        warp_batch_inverse(inv, okv, 3 * (m / 2));
        fe c1;
        ed::load_const(c1, ed::kC1);
        for (int q = 0; q < m / 2; ++q) {
            fe cy;
            if (okv[3 * q]) fq::mul(cy, c1, inv[3 * q]);   // c1 / y
            for (int h = 0; h < 2; ++h) {
                const int j = 2 * q + h;
                ok[j] = okv[3 * q] && okv[3 * q + 1 + h];
                if (!ok[j]) continue;
                fe a, d;
                fq::add(a, xs[j], one);
                fq::mul(xe[j], a, cy);                        // c1 a / y
                fq::sub(d, a, sp);
                fq::mul(ye[j], d, inv[3 * q + 1 + h]);        // (a - s) / (a + s)
            }
        }
        return;
    }
    fe xs[kEdChunk], ys[kEdChunk], den[kEdChunk];
    for (int j = 0; j < m; ++j) {
        glv_source(xs[j], ys[j], in, i0 + j, n, np);
        ok[j] = !(fq::is_zero_raw(xs[j]) && fq::is_zero_raw(ys[j]));
        fe a, apl;
        fq::add(a, xs[j], one);
        fq::add(apl, a, sp);
        fq::mul(den[j], ys[j], apl);
        ok[j] = ok[j] && !fq::is_zero(den[j]);
    }
    warp_batch_inverse(den, ok, m);
    for (int j = 0; j < m; ++j) {
        if (!ok[j]) continue;
        fe c, a;
        fq::add(a, xs[j], one);
        fq::add(c, a, sp);                  // a + s
        fq::mul(xe[j], a, c);
        ed::load_const(c, ed::kC1);
        fq::mul(xe[j], xe[j], c);
        fq::mul(xe[j], xe[j], den[j]);      // c1 a (a + s) / D
        fq::sub(c, a, sp);                  // a - s
        fq::mul(ye[j], c, ys[j]);
        fq::mul(ye[j], ye[j], den[j]);      // (a - s) y / D
    }
}

__device__ __forceinline__ void store_ed_stored(uint4* o, fe x, fe y) {
    fe u, k;
    ed::load_const(k, ed::kK);
    fq::mul(u, x, y);
    fq::mul(u, u, k);
    fq::canon(x, x);
    fq::canon(y, y);
    fq::canon(u, u);
    store_fe(o, x);
    store_fe(o + 3, y);
    store_fe(o + 6, u);
}

__device__ __forceinline__ void load_fe_cg(fe& a, const uint4* p) {   // through L2 (written by this thread)
    const uint4 u0 = __ldcg(p), u1 = __ldcg(p + 1), u2 = __ldcg(p + 2);
    a.v[0] = u0.x; a.v[1] = u0.y; a.v[2] = u0.z; a.v[3] = u0.w;
    a.v[4] = u1.x; a.v[5] = u1.y; a.v[6] = u1.z; a.v[7] = u1.w;
    a.v[8] = u2.x; a.v[9] = u2.y; a.v[10] = u2.z; a.v[11] = u2.w;
}

// s in standard form (the integer s, which is s / R as a Montgomery residue).
__device__ __constant__ static const uint32_t kSStd[fq::N] = {
    0xd09adc01u, 0x9c05824au, 0x0e1c7a7cu, 0x2e6bb28fu, 0xfc166427u, 0x2fe2cb65u,
    0x183465a4u, 0x86ef0d33u, 0x15ccbf8eu, 0x59416eceu, 0x062d349eu, 0x0032d756u};

__device__ __forceinline__ void add_one_raw(fe& r, const fe& a) {  // a + the integer 1
    fe o;
    fq::set_zero(o);
    o.v[0] = 1;
    fq::add(r, a, o);
}

__device__ __forceinline__ fe cst(const uint32_t (&c)[fq::N]) {
    fe r;
    ed::load_const(r, c);
    return r;
}

__device__ __forceinline__ fe mont_one() {
    fe r;
    fq::set_one(r);
    return r;
}

// Blocks of 128 per SM for the Edwards preparation: the GLV form at four (128
// registers, a few spills), the single-row form at two (its measured best, 0.485 ms for
// 2^20 points).
constexpr int prep_blocks_per_sm(bool glv) { return glv ? 4 : 2; }

// Stored Edwards rows of input points [a, b): row i, or rows 2i and 2i + 1 (P_i and
// phi(P_i) = (beta x_i, y_i)) with GLV. Same map as above, arranged to cost fewer
// multiplications and no local memory:
//  * The inputs stay in standard form. Read as Montgomery residues, x and y stand
//    for x / R and y / R; with the additive constants 1 and s entered in that same
//    scale (the integers 1 and s) every quantity the map divides is scaled by the
//    same power of R in numerator and denominator, so the Edwards coordinates come
//    out exact, in Montgomery form, with no conversion multiplications.
//  * GLV pair (P, phi(P)): one denominator t = y (a + s)(a' + s), a' = beta x + 1;
//    from t^-1 and u = y (a + s): 1/(a' + s) = t^-1 u, w = t^-1 (a' + s) = 1/u,
//    1/y = w (a + s), 1/(a + s) = w y; then x_e = c1 a / y, y_e = (a - s)/(a + s)
//    per row. Single row: t = y (a + s), x_e = c1 a (a + s) / t,
//    y_e = (a - s) y / t.
//  * A warp takes batches of 32 K consecutive points (lane l: points
//    base + 32 q + l, q < K) and inverts all their t with one field inversion
//    (Montgomery's trick over the lane's K points, warp_lane_inverse_wide over the
//    lanes). Pass 1 writes each point's prefix product and the values pass 2
//    needs into that point's own output rows; pass 2 reads them back (through
//    L2) and overwrites the rows with the stored form.
// A zero factor of t (the identity, or a point outside the map's domain) is
// replaced by 1 and the rows it feeds become the Edwards identity.
template <bool kGlv>
__global__ void __launch_bounds__(128, prep_blocks_per_sm(kGlv))
    k_prepare_ed(const uint4* __restrict__ in, uint4* out, size_t a, size_t b, int K) {
    __shared__ uint32_t mem[4][wred::kInverseWords];
    const int lane = threadIdx.x & 31;
    const size_t warp = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t per = 32 * (size_t)K;
    const size_t nb = (b - a + per - 1) / per;
    constexpr int kRows = kGlv ? 2 : 1;
    constexpr int kVec = ModelEdwards::kStored;  // uint4 per stored row
    for (size_t bt = warp; bt < nb; bt += warps) {
        const size_t base = a + bt * per + lane;
        fe acc = mont_one();
        for (int q = 0; q < K; ++q) {            // pass 1
            const size_t i = base + 32 * (size_t)q;
            if (i >= b) break;
            fe X, Y, A, D1, t;
            load_fe(X, in + 6 * i);
            load_fe(Y, in + 6 * i + 3);
            const bool id = fq::is_zero_raw(X) && fq::is_zero_raw(Y);
            add_one_raw(A, X);
            fq::add(D1, A, cst(kSStd));
            const bool okY = !id && !fq::is_zero(Y), ok1 = !id && !fq::is_zero(D1);
            const fe Yf = okY ? Y : mont_one(), D1f = ok1 ? D1 : mont_one();
            uint4* o = out + (size_t)kVec * kRows * i;
            fq::mul(t, Yf, D1f);
            if (kGlv) {
                fe BX, D2;
                fq::mul(BX, cst(kBeta), X);
                add_one_raw(D2, BX);
                fq::add(D2, D2, cst(kSStd));
                const bool ok2 = !id && !fq::is_zero(D2);
                store_fe(o + 6, t);              // u = y (a + s)
                store_fe(o + 9, BX);
                fq::mul(t, t, ok2 ? D2 : mont_one());
            }
            store_fe(o, acc);                    // prefix product
            store_fe(o + 3, t);
            fq::mul(acc, acc, t);
        }
        fe inv = warp_lane_inverse_wide(acc, mem[threadIdx.x >> 5]);   // acc^-1 on every lane
        for (int q = K - 1; q >= 0; --q) {       // pass 2
            const size_t i = base + 32 * (size_t)q;
            if (i >= b) continue;
            uint4* o = out + (size_t)kVec * kRows * i;
            fe X, Y, A, D1, pre, t, tinv;
            load_fe(X, in + 6 * i);
            load_fe(Y, in + 6 * i + 3);
            load_fe_cg(pre, o);
            load_fe_cg(t, o + 3);
            fq::mul(tinv, inv, pre);             // t^-1
            fq::mul(inv, inv, t);                // (prefix)^-1 for the next q down
            const bool id = fq::is_zero_raw(X) && fq::is_zero_raw(Y);
            add_one_raw(A, X);
            fq::add(D1, A, cst(kSStd));
            const bool okY = !id && !fq::is_zero(Y), ok1 = !id && !fq::is_zero(D1);
            if (kGlv) {
                fe u, BX, A2, D2, i2, w, iy, i1, cy;
                load_fe_cg(u, o + 6);
                load_fe_cg(BX, o + 9);
                add_one_raw(A2, BX);
                fq::add(D2, A2, cst(kSStd));
                const bool ok2 = !id && !fq::is_zero(D2);
                fq::mul(i2, tinv, u);                        // 1 / (a' + s)
                fq::mul(w, tinv, ok2 ? D2 : mont_one());     // 1 / (y (a + s))
                fq::mul(iy, w, ok1 ? D1 : mont_one());       // 1 / y
                fq::mul(i1, w, okY ? Y : mont_one());        // 1 / (a + s)
                fq::mul(cy, cst(ed::kC1), iy);               // c1 / y
                fe xe, ye, d;
                if (okY && ok1) {
                    fq::mul(xe, A, cy);
                    fq::sub(d, A, cst(kSStd));
                    fq::mul(ye, d, i1);
                    store_ed_stored(o, xe, ye);
                } else {
                    store_ed_identity(o);
                }
                if (okY && ok2) {
                    fq::mul(xe, A2, cy);
                    fq::sub(d, A2, cst(kSStd));
                    fq::mul(ye, d, i2);
                    store_ed_stored(o + kVec, xe, ye);
                } else {
                    store_ed_identity(o + kVec);
                }
            } else {
                if (okY && ok1) {
                    fe ct, xe, ye, d;
                    fq::mul(ct, cst(ed::kC1), tinv);         // c1 / t
                    fq::mul(xe, A, D1);
                    fq::mul(xe, xe, ct);                     // c1 a (a + s) / t
                    fq::sub(d, A, cst(kSStd));
                    fq::mul(ye, d, Y);
                    fq::mul(ye, ye, tinv);                   // (a - s) y / t
                    store_ed_stored(o, xe, ye);
                } else {
                    store_ed_identity(o);
                }
            }
        }
    }
}

// Fixed-base precomputation for resident Edwards sets: row q Wd + j of out is the
// stored form of 2^(c j) P'_q for j < Wd, P' the np stored points of the
// standard-form input (point-major, so the rows of a contiguous range of points are
// contiguous). Each lane maps its chunk to Edwards, then doubles it c times per
// window and normalises it with one inversion per warp and window. With these,
// every window of an MSM adds into the same buckets:
// sum_j 2^(cj) sum_b b B_jb = sum_b b sum_j B'_jb with B' over the shifted points.
__global__ void __launch_bounds__(128, 3) k_precompute_ed(const uint4* __restrict__ in, uint4* __restrict__ out,
                                                       size_t n, size_t np, int c, int Wd) {
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const size_t i0 = t * kEdChunk;
    const int m = i0 >= np ? 0 : (int)(np - i0 < (size_t)kEdChunk ? np - i0 : (size_t)kEdChunk);
    fe den[kEdChunk];
    bool ok[kEdChunk];
    ed::ext P[kEdChunk];
    {
        fe xe[kEdChunk], ye[kEdChunk];
        ed_affine_chunk(in, n, np, i0, m, np != n && (np & 1) == 0, xe, ye, ok);  // rows [0, np): launch-wide
        for (int q = 0; q < m; ++q) {
            uint4* o = out + (size_t)ModelEdwards::kStored * ((i0 + q) * (size_t)Wd);
            if (ok[q]) {
                ed::stored Q;
                Q.x = xe[q];
                Q.y = ye[q];
                ed::from_stored(P[q], Q);   // u unused by from_stored
                store_ed_stored(o, xe[q], ye[q]);
            } else {
                ed::set_inf(P[q]);          // the identity stays the identity
                store_ed_identity(o);
            }
        }
    }
    for (int j = 1; j < Wd; ++j) {
        for (int q = 0; q < m; ++q) {
            for (int d = 0; d < c; ++d) ed::dbl(P[q]);
            den[q] = P[q].Z;
            ok[q] = !fq::is_zero(P[q].Z);
        }
        warp_batch_inverse(den, ok, m);
        for (int q = 0; q < m; ++q) {
            uint4* o = out + (size_t)ModelEdwards::kStored * ((i0 + q) * (size_t)Wd + j);
            if (!ok[q]) {
                store_ed_identity(o);
                continue;
            }
            fe x, y;
            fq::mul(x, P[q].X, den[q]);
            fq::mul(y, P[q].Y, den[q]);
            store_ed_stored(o, x, y);
        }
    }
}

// ---------------------------------------------------------------- stage 2

// Window digits of one scalar (8 words, little-endian) for point index `idx`:
// |digit| (0 = no contribution) with its sign in bit 31, window-major ([W][np]). The
// point of an item follows from its place (item_point), so it is not stored. Returns how
// many digits are not zero (kCount; else 0).
template <bool kCount>
__device__ __forceinline__ uint32_t emit_digits(const uint32_t (&s)[8], int c, int W, int sgn, size_t idx,
                                            size_t np, uint32_t* __restrict__ keys) {
    const uint32_t cmask = (1u << c) - 1u, half = 1u << (c - 1);
    uint32_t carry = 0, nonzero = 0;
    for (int j = 0; j < W; ++j) {
        int b0 = j * c, w = b0 >> 5, off = b0 & 31;
        uint32_t raw = 0;
        if (w < 8) {
            raw = s[w] >> off;
            if (off + c > 32 && w + 1 < 8) raw |= s[w + 1] << (32 - off);
            raw &= cmask;
        }
        uint32_t key, neg = 0;
        if (sgn) {
            uint32_t v = raw + carry;
            if (v > half) {
                key = (1u << c) - v;  // |v - 2^c|
                neg = 1;
                carry = 1;
            } else {
                key = v;
                carry = 0;
            }
        } else {
            key = raw;
        }
        keys[(size_t)j * np + idx] = key | (neg << 31);
        if (kCount) nonzero += key != 0;
    }
    return nonzero;
}

constexpr uint32_t kSign = 0x80000000u;

// The stored point of item j of a window: point j, or with precomputed shifted points
// (one window of Wd np items, item j' np + i the digit j' of point i) the copy
// 2^(c j') P_i at row i Wd + j'. Wd = 0: no precomputed points.
__device__ __forceinline__ uint32_t item_point(size_t j, size_t np, int Wd) {
    if (Wd == 0) return (uint32_t)j;
    const uint32_t d = (uint32_t)(j / np), i = (uint32_t)(j - (size_t)d * np);
    return i * (uint32_t)Wd + d;
}

// GLV split of a scalar k < 2^256: k mod r = k1 + lambda k2 with 0 <= k1 < lambda
// and k2 <= lambda + 1 (both below 2^127), lambda = x0^2 - 1 and
// lambda^2 + lambda + 1 = r. k is first reduced below r by conditional
// subtraction of 8r, 4r, 2r, r (2^256 < 16 r). Then q = floor(k mu / 2^256) with
// mu = floor(2^256 / lambda) is k2 or k2 - 1 (k mu / 2^256 > k / lambda - 1 since
// k < 2^256), fixed by one conditional subtraction of lambda.
__device__ __constant__ static const uint32_t kR8[4][8] = {
    {0x00000008u, 0x508c0000u, 0x80000008u, 0xcd53b7f6u, 0xe1bd800au, 0x05a268f2u, 0xd1652ab3u, 0x955b2af4u},
    {0x00000004u, 0x28460000u, 0x40000004u, 0x66a9dbfbu, 0x70dec005u, 0x82d13479u, 0x68b29559u, 0x4aad957au},
    {0x00000002u, 0x14230000u, 0xa0000002u, 0xb354edfdu, 0xb86f6002u, 0xc1689a3cu, 0x34594aacu, 0x2556cabdu},
    {0x00000001u, 0x0a118000u, 0xd0000001u, 0x59aa76feu, 0x5c37b001u, 0x60b44d1eu, 0x9a2ca556u, 0x12ab655eu}};
__device__ __constant__ static const uint32_t kLambda[4] = {0x00000000u, 0x0a118000u, 0x90000001u, 0x452217ccu};
__device__ __constant__ static const uint32_t kMu[5] = {0xaf90182cu, 0x7f72ed32u, 0x9fd37160u, 0xb3f7aa96u,
                                                        0x00000003u};

__device__ __forceinline__ void glv_split(uint32_t (&k)[8], uint32_t (&k1)[8], uint32_t (&k2)[8]) {
    for (int m = 0; m < 4; ++m) {  // k -= 8r, 4r, 2r, r where k is at least that
        uint32_t d[8];
        uint64_t borrow = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            uint64_t t = (uint64_t)k[w] - kR8[m][w] - borrow;
            d[w] = (uint32_t)t;
            borrow = (t >> 63) & 1u;
        }
        if (!borrow) {
#pragma unroll
            for (int w = 0; w < 8; ++w) k[w] = d[w];
        }
    }
    // q = floor(k mu / 2^256): columns 8..12 of the 8 x 5 word product
    uint32_t prod[13];
#pragma unroll
    for (int w = 0; w < 13; ++w) prod[w] = 0;
    for (int i = 0; i < 8; ++i) {
        uint64_t carry = 0;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            uint64_t t = (uint64_t)k[i] * kMu[j] + prod[i + j] + carry;
            prod[i + j] = (uint32_t)t;
            carry = t >> 32;
        }
        for (int w = i + 5; w < 13 && carry; ++w) {
            uint64_t t = (uint64_t)prod[w] + carry;
            prod[w] = (uint32_t)t;
            carry = t >> 32;
        }
    }
    uint32_t q[4] = {prod[8], prod[9], prod[10], prod[11]};  // k mu < 2^383, so prod[12] = 0
    // rem = k - q lambda (fits in 5 words: rem < 2 lambda < 2^128)
    uint32_t ql[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) ql[w] = 0;
    for (int i = 0; i < 4; ++i) {
        uint64_t carry = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint64_t t = (uint64_t)q[i] * kLambda[j] + ql[i + j] + carry;
            ql[i + j] = (uint32_t)t;
            carry = t >> 32;
        }
        ql[i + 4] = (uint32_t)carry;
    }
    uint32_t rem[8];
    uint64_t borrow = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint64_t t = (uint64_t)k[w] - ql[w] - borrow;
        rem[w] = (uint32_t)t;
        borrow = (t >> 63) & 1u;
    }
    // rem >= lambda ? (rem < 2^128 here, so words 4..7 are zero)
    bool ge = true;
    for (int w = 3; w >= 0; --w) {
        if (rem[w] != kLambda[w]) {
            ge = rem[w] > kLambda[w];
            break;
        }
    }
    if (rem[4] | rem[5] | rem[6] | rem[7]) ge = true;
    if (ge) {
        uint64_t br = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            uint64_t t = (uint64_t)rem[w] - (w < 4 ? kLambda[w] : 0u) - br;
            rem[w] = (uint32_t)t;
            br = (t >> 63) & 1u;
        }
        uint64_t cy = 1;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint64_t t = (uint64_t)q[w] + cy;
            q[w] = (uint32_t)t;
            cy = t >> 32;
        }
    }
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        k1[w] = w < 4 ? rem[w] : 0u;
        k2[w] = w < 4 ? q[w] : 0u;
    }
}

// The digits of scalar i; returns how many are not zero (kCount; else 0).
template <bool kCount>
__device__ __forceinline__ uint32_t scalar_digits(const uint4* __restrict__ scalars, size_t i, size_t n, int c, int W, int sgn,
                                                  int bits, int glv, uint32_t* __restrict__ keys, int* __restrict__ status) {
    uint4 lo = scalars[2 * i], hi = scalars[2 * i + 1];
    uint32_t s[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    if (bits < 256) {
        uint32_t over = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            int lo_bit = 32 * k;
            uint32_t m = lo_bit >= bits ? 0xffffffffu
                         : (bits - lo_bit >= 32 ? 0u : ~((1u << (bits - lo_bit)) - 1u));
            over |= s[k] & m;
        }
        if (over) atomicCAS(status, 0, MSM377_ERANGE);   // the first error of the call stays
    }
    if (!glv) return emit_digits<kCount>(s, c, W, sgn, i, n, keys);
    uint32_t k1[8], k2[8];
    glv_split(s, k1, k2);
    const uint32_t m = emit_digits<kCount>(k1, c, W, sgn, 2 * i, 2 * n, keys);     // P_i
    return m + emit_digits<kCount>(k2, c, W, sgn, 2 * i + 1, 2 * n, keys);         // phi(P_i)
}

// kCount: the count of digits that are not zero is added to *nonzero (piece_cap), 5 us at
// n = 2^20; calls of short pieces, which do not ask for it, are spared 1 us of 8.
constexpr int kDigitThreads = 256;

template <bool kCount>
__global__ void __launch_bounds__(kDigitThreads) k_digits(const uint4* __restrict__ scalars, size_t n, int c, int W, int sgn,
                                                          int bits, int glv, uint32_t* __restrict__ keys,
                                                          int* __restrict__ status, uint32_t* __restrict__ nonzero) {
    __shared__ uint32_t block_count;
    const size_t i = blockIdx.x * (size_t)kDigitThreads + threadIdx.x;
    uint32_t m = i < n ? scalar_digits<kCount>(scalars, i, n, c, W, sgn, bits, glv, keys, status) : 0u;
    if (!kCount) return;
    if (threadIdx.x == 0) block_count = 0;
    __syncthreads();
    m = __reduce_add_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicAdd(&block_count, m);
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(nonzero, block_count);
}

// ---------------------------------------------------------------- stage 3: radix sort

// Digits of RB bits per pass, R = 2^RB bins (the library sorts 8 bits per pass).
template <int RB>
__global__ void k_sort_hist(const uint32_t* __restrict__ keys, size_t n, int shift, size_t tiles,
                            uint32_t* __restrict__ hist) {
    constexpr int R = 1 << RB;
    __shared__ uint32_t cnt[R];
    const size_t t = blockIdx.x, w = blockIdx.y;
    for (int d = threadIdx.x; d < R; d += kSortThreads) cnt[d] = 0;
    __syncthreads();
    const uint32_t* seg = keys + w * n;
    const size_t start = t * kSortTile;
#pragma unroll
    for (int e = 0; e < kSortItems; ++e) {
        size_t idx = start + (size_t)e * kSortThreads + threadIdx.x;
        if (idx < n) atomicAdd(&cnt[(seg[idx] >> shift) & (R - 1)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < R; d += kSortThreads) hist[(w * R + d) * tiles + t] = cnt[d];
}

// Exclusive block-wide scan of one value per thread (256 threads).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
    __shared__ uint32_t warp_sums[kSortThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < kSortThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kSortThreads / 32) warp_sums[lane] = s;
    }
    __syncthreads();
    uint32_t before = wid ? warp_sums[wid - 1] : 0;
    if (total) *total = warp_sums[kSortThreads / 32 - 1];
    __syncthreads();
    return before + x - v;
}

// For each (window, digit): exclusive scan over tiles in place; the digit total goes to dtot.
template <int RB>
__global__ void k_sort_scan_tiles(uint32_t* __restrict__ hist, size_t tiles, uint32_t* __restrict__ dtot) {
    constexpr int R = 1 << RB;
    const size_t d = blockIdx.x, w = blockIdx.y;
    uint32_t* row = hist + (w * R + d) * tiles;
    const size_t per = (tiles + kSortThreads - 1) / kSortThreads;
    const size_t lo = threadIdx.x * per;
    uint32_t local = 0;
    for (size_t k = 0; k < per; ++k)
        if (lo + k < tiles) local += row[lo + k];
    uint32_t total;
    uint32_t run = block_exclusive_scan(local, &total);
    for (size_t k = 0; k < per; ++k) {
        if (lo + k < tiles) {
            uint32_t c = row[lo + k];
            row[lo + k] = run;
            run += c;
        }
    }
    if (threadIdx.x == 0) dtot[w * R + d] = total;
}

// Exclusive scan of the R digit totals of a window (R / 256 consecutive digits per thread).
template <int RB>
__global__ void k_sort_scan_digits(uint32_t* __restrict__ dtot) {
    constexpr int R = 1 << RB, PER = R / kSortThreads;
    uint32_t* row = dtot + blockIdx.x * R + threadIdx.x * PER;
    uint32_t v[PER], local = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = row[k];
        local += v[k];
    }
    uint32_t run = block_exclusive_scan(local, nullptr);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        row[k] = run;
        run += v[k];
    }
}

template <int RB>
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, size_t n, int shift, size_t tiles,
    const uint32_t* __restrict__ hist, const uint32_t* __restrict__ doff, size_t np, int Wd) {
    constexpr int R = 1 << RB;
    __shared__ uint32_t wcnt[kSortThreads / 32][R];
    __shared__ uint32_t base[R];
    const size_t t = blockIdx.x, w = blockIdx.y;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < (kSortThreads / 32) * R; k += kSortThreads)
        (&wcnt[0][0])[k] = 0;
    __syncthreads();
    const uint32_t lt_mask = (1u << lane) - 1u;
    const size_t seg = w * n;
    const size_t sub = t * kSortTile + (size_t)wid * (32 * kSortItems);
    uint32_t key[kSortItems], val[kSortItems], dig[kSortItems], rank[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        size_t idx = sub + (size_t)r * 32 + lane;
        bool valid = idx < n;
        key[r] = valid ? kin[seg + idx] : 0u;
        if (vin) {
            val[r] = valid ? vin[seg + idx] : 0u;
        } else {        // the first pass: the item's point and sign
            val[r] = item_point(idx, np, Wd) | (key[r] & kSign);
            key[r] &= ~kSign;
        }
        // Items past the end sort last in the tile and are never written.
        dig[r] = valid ? ((key[r] >> shift) & (R - 1)) : (R - 1);
        uint32_t peers = __match_any_sync(0xffffffffu, dig[r]);
        uint32_t before = wcnt[wid][dig[r]];
        __syncwarp();
        if (lane == __ffs(peers) - 1) wcnt[wid][dig[r]] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt_mask);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < R; d += kSortThreads) {
        uint32_t run = 0;
#pragma unroll
        for (int k = 0; k < kSortThreads / 32; ++k) {
            uint32_t c = wcnt[k][d];
            wcnt[k][d] = run;
            run += c;
        }
        base[d] = doff[w * R + d] + hist[(w * R + d) * tiles + t];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        size_t idx = sub + (size_t)r * 32 + lane;
        if (idx < n) {
            size_t pos = (size_t)base[dig[r]] + wcnt[wid][dig[r]] + rank[r];
            if (pos < n) {  // always true when the counts agree; keeps writes in bounds
                kout[seg + pos] = key[r];
                vout[seg + pos] = val[r];
            }
        }
    }
}

// Run starts of the sorted keys: start[w nb + k] = w n + the first position in window
// w with key >= k, for k < nb (the bin offsets that the counting sort has anyway). Item j
// writes the keys above the item before it up to its own, and the last item the keys above
// its own. Where digits leave many keys out, such a range can be a whole window's keys:
// ranges of more than kWideGap are written by the block together (13 windows of 2^19 keys,
// 100 zero scalars, c = 20: by one thread each 1745 us).
constexpr int kStartThreads = 256;
constexpr uint32_t kWideGap = 16;

__global__ void __launch_bounds__(kStartThreads) k_run_starts(const uint32_t* __restrict__ keys, size_t n, uint32_t nb,
                                                              uint32_t* __restrict__ start) {
    __shared__ uint3 wide[kStartThreads + 1];   // {first key, end, value}
    __shared__ uint32_t nwide;
    if (threadIdx.x == 0) nwide = 0;
    __syncthreads();
    const size_t j = blockIdx.x * (size_t)kStartThreads + threadIdx.x;
    const size_t w = blockIdx.y;
    const uint32_t* kw = keys + w * n;
    uint32_t* row = start + w * nb;
    auto fill = [&](uint32_t lo, uint32_t end, uint32_t value) {
        if (end > nb) end = nb;   // keys are below nb by construction
        if (end > lo && end - lo > kWideGap) {
            wide[atomicAdd(&nwide, 1u)] = make_uint3(lo, end, value);
            return;
        }
        for (uint32_t k = lo; k < end; ++k) row[k] = value;
    };
    if (j < n) {
        const uint32_t key = kw[j];
        fill(j ? kw[j - 1] + 1 : 0u, key + 1, (uint32_t)(w * n + j));
        if (j + 1 == n) fill(key + 1, nb, (uint32_t)((w + 1) * n));
    }
    __syncthreads();
    for (uint32_t i = 0; i < nwide; ++i) {
        const uint3 r = wide[i];
        for (uint32_t k = r.x + threadIdx.x; k < r.y; k += kStartThreads) row[k] = r.z;
    }
}

// ---------------------------------------------------------------- stage 3 (counting sort)
//
// Bucket order by counting: every (window, key) is a bin; one pass counts the
// items of each bin with warp-aggregated atomics, a scan turns the counts into
// bin offsets (window w's bins start at w np, since each window holds np items),
// and one pass scatters every item to its bin's next free slot. The order inside
// a bin is not kept -- it does not matter, since a bucket's sum is the same group
// element in any order. Two passes over the keys instead of a
// histogram and a scatter pass per 8 key bits.
constexpr int kScanBlock = 1024, kScanPer = 4, kScanTile = kScanBlock * kScanPer;

// Grid (items of a window / 256, windows): item i = w np + j of window w = blockIdx.y.
// Counts per (window, key) bin; each item keeps its rank among the items of its bin
// (the warp's share from one atomic per distinct bin, then the lanes' order), so the
// scatter needs no atomics. This global-counter form serves key ranges too wide for
// the shared-memory tiles below (c >= 18 with signed digits, c >= 17 unsigned).
__global__ void k_bin_count(const uint32_t* __restrict__ keys, size_t np, uint32_t nb,
                            uint32_t* __restrict__ counts, uint32_t* __restrict__ rank) {
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const bool valid = j < np;
    const size_t i = (size_t)blockIdx.y * np + j;
    const uint32_t bin = valid ? blockIdx.y * nb + (keys[i] & ~kSign) : 0xffffffffu;
    const uint32_t peers = __match_any_sync(0xffffffffu, bin);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (valid && lane == leader) base = atomicAdd(&counts[bin], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (valid) rank[i] = base + __popc(peers & ((1u << lane) - 1u));
}
__global__ void __launch_bounds__(kScanBlock) k_scan_tiles(uint32_t* __restrict__ x, size_t m,
                                                           uint32_t* __restrict__ bsum) {
    __shared__ uint32_t warp_tot[kScanBlock / 32];
    const size_t base = (size_t)blockIdx.x * kScanTile + (size_t)threadIdx.x * kScanPer;
    uint32_t v[kScanPer], local = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = base + k < m ? x[base + k] : 0u;
        local += v[k];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t inc = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;  // inclusive over warps
    }
    __syncthreads();
    uint32_t run = inc - local + (wid ? warp_tot[wid - 1] : 0u);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (base + k < m) x[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == kScanBlock - 1) bsum[blockIdx.x] = warp_tot[kScanBlock / 32 - 1];
}

// Exclusive scan of the tile totals in one block (any count: a serial run per thread).
__global__ void __launch_bounds__(kScanBlock) k_scan_totals(uint32_t* __restrict__ bsum, size_t nb) {
    __shared__ uint32_t warp_tot[kScanBlock / 32];
    const size_t per = (nb + kScanBlock - 1) / kScanBlock;
    const size_t lo = threadIdx.x * per;
    uint32_t local = 0;
    for (size_t k = lo; k < lo + per && k < nb; ++k) local += bsum[k];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t inc = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    uint32_t run = inc - local + (wid ? warp_tot[wid - 1] : 0u);
    for (size_t k = lo; k < lo + per && k < nb; ++k) {
        const uint32_t c = bsum[k];
        bsum[k] = run;
        run += c;
    }
}

__global__ void k_scan_add(uint32_t* __restrict__ x, size_t m, const uint32_t* __restrict__ bsum) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < m) x[i] += bsum[i / kScanTile];
}

// Each item's point and sign to its slot: the bin's offset plus its rank in the bin.
__global__ void k_bin_scatter(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ rank,
                              uint32_t* __restrict__ out, size_t total, size_t items, uint32_t nb,
                              const uint32_t* __restrict__ start, size_t np, int Wd) {
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (j >= items) return;
    const size_t i = (size_t)blockIdx.y * items + j;
    const uint32_t key = kin[i];
    const size_t pos = (size_t)start[blockIdx.y * nb + (key & ~kSign)] + rank[i];
    if (pos < total) out[pos] = item_point(j, np, Wd) | (key & kSign);  // in bounds when the counts agree
}

// The same counting sort with the counts taken per tile in shared memory, for key
// ranges whose counters fit there (no global atomics at all). Tile t of window w
// holds items [t T, (t + 1) T); its block counts the tile's keys in 16-bit shared
// counters packed two to a word (T < 2^16, so no count reaches the neighbour's
// half) and gives each item its rank among the tile's items of the same key. The
// tile counts go to cnt[w][t][key]; a column pass (k_tile_totals) sums them into the bin
// totals, scans these within blocks of bins and counts the pieces they will be cut into;
// a second one (k_tile_offsets) adds the earlier blocks' totals, which gives each (window,
// key) its offset, and turns cnt into each tile's first slot per key (offset + counts of
// the earlier tiles); an item's slot is that plus its rank.
constexpr int kTileThreads = 1024;
constexpr uint32_t kTileItemsMax = 65535;
constexpr size_t kTileSmemMax = 200 * 1024;    // packed counters of one block (GB300: 227 KB opt-in)

// Grid (tiles, windows). Plain shared atomics: with random keys the counters rarely
// collide. Measured on GB300 (n = 2^20, c = 16): one atomic per distinct key and
// warp (found with match.any) made the head 0.09 ms slower with random scalars, and a
// one-atomic path for warps whose keys are all equal moved it by at most 0.02 ms
// with all-equal scalars.
__global__ void __launch_bounds__(kTileThreads) k_tile_count(const uint32_t* __restrict__ keys, size_t np,
                                                             uint32_t nb, uint32_t T, uint32_t ntiles,
                                                             uint32_t* __restrict__ cnt, uint32_t* __restrict__ rank) {
    extern __shared__ uint32_t h[];
    const uint32_t hw = (nb + 1) / 2;
    for (uint32_t k = threadIdx.x; k < hw; k += blockDim.x) h[k] = 0;
    __syncthreads();
    const size_t w = blockIdx.y;
    const size_t lo = (size_t)blockIdx.x * T;
    const size_t hi = lo + T < np ? lo + T : np;
    const uint32_t* kw = keys + w * np;
    uint32_t* rw = rank + w * np;
    for (size_t j = lo + threadIdx.x; j < hi; j += blockDim.x) {
        const uint32_t key = kw[j] & ~kSign;
        if (key >= nb) continue;   // keys are below nb by construction
        const uint32_t sh = (key & 1u) << 4;
        const uint32_t old = atomicAdd(&h[key >> 1], 1u << sh);
        rw[j] = (old >> sh) & 0xffffu;
    }
    __syncthreads();
    uint32_t* cw = cnt + (w * ntiles + blockIdx.x) * nb;
    for (uint32_t k = threadIdx.x; k < nb; k += blockDim.x) cw[k] = (h[k >> 1] >> ((k & 1u) << 4)) & 0xffffu;
}

// Grid (items of a window / 256, windows): each item to its tile's slot for the key
// plus its rank.
__global__ void k_tile_scatter(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ rank,
                               uint32_t* __restrict__ out, size_t total, size_t items, uint32_t nb, uint32_t T,
                               uint32_t ntiles, const uint32_t* __restrict__ cnt, size_t np, int Wd) {
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (j >= items) return;
    const size_t w = blockIdx.y;
    const size_t i = w * items + j;
    const uint32_t key = kin[i], bin = key & ~kSign;
    if (bin >= nb) return;
    const size_t t = j / T;
    const size_t pos = (size_t)cnt[(w * ntiles + t) * nb + bin] + rank[i];
    if (pos < total) out[pos] = item_point(j, np, Wd) | (key & kSign);
}

// ---------------------------------------------------------------- stages 4-5
//
// A bucket's run of m sorted items is cut into ceil(m / cap) pieces of nearly equal
// length. Pieces are listed by length, longest first (a counting sort over the at most
// kMaxPiece lengths), and one thread sums one piece: the lanes of a warp then start,
// add and store together, where threads over equal chunks of the sorted stream spent
// a tenth of their additions on lanes waiting for another lane's run end, and every
// run crossing a chunk edge cost a full addition to put together. Measured at
// n = 2^20: accumulation and merges 5742 + 420 -> 5570 + 120 us (XYZZ, c = 16),
// 4179 + 424 -> 3740 + 75 us (Edwards + GLV, c = 17); both now run the multiply pipe at 0.9
// to 0.96 of its measured peak.
// A bucket of one piece gets its sum directly. The pieces of any other leave partial
// sums in consecutive slots, put together by k_merge_parts: a few by one thread in
// sequence, more by blocks that sum up to kTreeParts each in a tree of
// four-lane additions, in up to three levels -- so a bucket that holds a whole window
// (all-equal scalars, a nearly empty top window) costs O(log) sequential additions.
constexpr uint32_t kMaxPiece = 256;     // longest piece a plan may ask for
constexpr uint32_t kTreeParts = 64;
constexpr uint32_t kPart = 0x80000000u; // destination is a partial-sum slot, not a bucket
constexpr int kPieceThreads = 256;

// Device counters of one window group, zeroed before use. Indices into uint32_t words.
enum : uint32_t { kHist = 0, kCursor = kMaxPiece + 1, kNParts = 2 * (kMaxPiece + 1), kNSmall, kNTree /* 3 levels */,
                  kNonzero = kNTree + 3 /* the first group's: digits of all groups */,
                  kCtrlWords = (kNonzero + 1 + 31) / 32 * 32 };

struct PieceArgs {
    const uint32_t* start;  // first item of each bin (w, key), key < nb; the next bin's start ends it
    uint32_t nb, Bp;
    int w0, nwin;           // windows of this group
    uint32_t total;         // all windows' items: the end of the last bin
    uint32_t cap;           // longest piece where most digits are nonzero (piece_cap)
    uint32_t cap_few;       // and the shortest that it may become where few are
    const uint32_t* nonzero;   // digits that are not zero, over all windows (null: cap as it is)
    uint32_t all;           // items of all windows
    uint32_t group_items;   // items of a full group
    uint32_t wave;          // resident threads
    uint32_t shared;        // half a thread's share of the whole batch's items (0: a single call)
    int levels;             // tree levels of the merge that are launched
    uint32_t small_parts;   // buckets of up to this many parts are summed by one thread
    uint32_t* ctrl;
    uint4* pieces;          // {first item, length, destination, -}
    uint4* small;           // {first part, parts, destination, -}
    uint4* tree[3];
    uint4* buckets;
};

struct BinRun {
    uint32_t s, m, bucket;
};

// Bin id (over the group's windows) -> its run; m = 0 and no bucket for key 0 (zero
// digits) and past the end.
__device__ __forceinline__ BinRun bin_run(const PieceArgs& a, size_t id) {
    BinRun r = {0, 0, kNone};
    if (id >= (size_t)a.nwin * a.nb) return r;
    const uint32_t wi = (uint32_t)(id / a.nb), key = (uint32_t)(id - (size_t)wi * a.nb);
    const size_t g = (size_t)(a.w0 + wi) * a.nb + key;
    r.s = a.start[g];
    // bins are contiguous over all windows; the last one ends at the last item
    const uint32_t e = (wi + 1 == (uint32_t)a.nwin && key + 1 == a.nb) ? a.total : a.start[g + 1];
    if (key == 0) return r;
    r.m = e - r.s;
    r.bucket = (uint32_t)(a.w0 + wi) * a.Bp + key - 1;
    return r;
}

// The longest piece. cap takes every digit for nonzero, but a thread's share is of those
// that are: 2^20 scalars of one, c = 12, Edwards + GLV, are one run of 2^20 points among 23
// million zero digits, and in pieces of cap = 256 it kept 4096 threads for 1925 us. With
// fewer than half the digits nonzero the piece is a thread's share of them (plus 4, as in
// make_plan), but no shorter than cap_few, nor so short that the pieces of the nonzero digits
// outgrow the bound group_items / cap on which the lists are sized.
__device__ __forceinline__ uint32_t piece_cap(const PieceArgs& a) {
    if (!a.nonzero) return a.cap;
    const uint32_t nz = *a.nonzero;
    if (nz >= a.all / 2) return a.cap;
    const uint32_t bound = (uint32_t)(((uint64_t)nz * a.cap + a.group_items - 1) / a.group_items);
    uint32_t k = nz / a.wave + 5;
    const uint32_t shared = (uint32_t)((uint64_t)nz * a.shared / a.all);
    if (k < shared) k = shared;
    if (k < bound) k = bound;
    if (k < a.cap_few) k = a.cap_few;
    return k < a.cap ? k : a.cap;
}

// The pieces of a run of m items, counted by length.
__device__ __forceinline__ void count_pieces(uint32_t* h, uint32_t m, uint32_t cap) {
    const uint32_t np = (m + cap - 1) / cap, q = m / np, big = m - q * np;
    if (big) atomicAdd(&h[q + 1], big);
    atomicAdd(&h[q], np - big);
}

__global__ void __launch_bounds__(kPieceThreads) k_piece_count(PieceArgs a) {
    __shared__ uint32_t h[kMaxPiece + 1];
    for (uint32_t k = threadIdx.x; k <= kMaxPiece; k += kPieceThreads) h[k] = 0;
    __syncthreads();
    const BinRun r = bin_run(a, blockIdx.x * (size_t)kPieceThreads + threadIdx.x);
    if (r.m) count_pieces(h, r.m, piece_cap(a));
    __syncthreads();
    for (uint32_t k = threadIdx.x; k <= a.cap; k += kPieceThreads)
        if (h[k]) atomicAdd(&a.ctrl[kHist + k], h[k]);
}

// Counting sort by tiles, after k_tile_count. Thread (w, key): bins[w][key] <- the counts of
// the block's earlier bins, bsum[block] <- the block's total, and the pieces of all bins
// counted by length (pieces = 0: not counted here, several window groups). What bounds
// these two kernels is the column reads (40 MB each way at n = 2^20, c = 16); small calls pay
// their launches, and one launch each for totals, scan of the tiles, scan of the totals,
// addition, piece counts and offsets was 10 to 15 us more than these two.
constexpr int kBinBlock = 1024;

__global__ void __launch_bounds__(kBinBlock) k_tile_totals(const uint32_t* __restrict__ cnt, uint32_t nb, uint32_t ntiles,
                                                          uint32_t W, uint32_t* __restrict__ bins,
                                                          uint32_t* __restrict__ bsum, PieceArgs a, int pieces) {
    __shared__ uint32_t h[kMaxPiece + 1];
    __shared__ uint32_t warp_tot[kBinBlock / 32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (t <= (int)kMaxPiece) h[t] = 0;
    __syncthreads();
    const size_t id = blockIdx.x * (size_t)kBinBlock + t;
    uint32_t m = 0;
    if (id < (size_t)W * nb) {
        const size_t w = id / nb, k = id - w * nb;
        const uint32_t* c = cnt + w * ntiles * nb + k;
        for (uint32_t u = 0; u < ntiles; ++u) m += c[(size_t)u * nb];
        if (pieces && k != 0 && m) count_pieces(h, m, piece_cap(a));
    }
    uint32_t x = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t y = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        warp_tot[lane] = y;   // inclusive over warps
    }
    __syncthreads();
    if (id < (size_t)W * nb) bins[id] = x - m + (wid ? warp_tot[wid - 1] : 0u);
    if (t == kBinBlock - 1) bsum[blockIdx.x] = warp_tot[kBinBlock / 32 - 1];
    if (pieces && t <= (int)a.cap && h[t]) atomicAdd(&a.ctrl[kHist + t], h[t]);
}

// Thread (w, key): bins[w][key] <- the bin's offset, and cnt[w][t][key] <- the slot of tile
// t's first item of that key, the offset plus the counts of tiles t' < t.
__global__ void __launch_bounds__(256) k_tile_offsets(uint32_t* __restrict__ cnt, uint32_t nb, uint32_t ntiles, uint32_t W,
                                                     uint32_t* __restrict__ bins, const uint32_t* __restrict__ bsum) {
    __shared__ uint32_t part[8];
    const int t = threadIdx.x;
    const uint32_t block = blockIdx.x / (kBinBlock / 256);   // the block of bins that this one is in
    uint32_t before = 0;
    for (uint32_t b = t; b < block; b += 256) before += bsum[b];
    before = __reduce_add_sync(0xffffffffu, before);
    if ((t & 31) == 0) part[t >> 5] = before;
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) run += part[k];
    const size_t id = blockIdx.x * (size_t)256 + t;
    if (id >= (size_t)W * nb) return;
    const size_t w = id / nb, k = id - w * nb;
    run += bins[id];
    bins[id] = run;
    uint32_t* c = cnt + w * ntiles * nb + k;
    constexpr uint32_t kStep = 16;   // loads in flight per thread
    for (uint32_t t0 = 0; t0 < ntiles; t0 += kStep) {
        uint32_t v[kStep];
#pragma unroll
        for (uint32_t u = 0; u < kStep; ++u) v[u] = t0 + u < ntiles ? c[(size_t)(t0 + u) * nb] : 0u;
#pragma unroll
        for (uint32_t u = 0; u < kStep; ++u) {
            if (t0 + u < ntiles) c[(size_t)(t0 + u) * nb] = run;
            run += v[u];
        }
    }
}

// Appends the merge work of a bucket cut into np pieces; returns its first part slot.
__device__ __forceinline__ uint32_t plan_merge(const PieceArgs& a, uint32_t np, uint32_t bucket) {
    // partial sums of the tree's inner levels; the last level launched takes what is left
    const uint32_t n1 = (np + kTreeParts - 1) / kTreeParts, n2 = (n1 + kTreeParts - 1) / kTreeParts;
    const uint32_t extra = np <= a.small_parts || n1 == 1 || a.levels == 1 ? 0 : (n2 == 1 || a.levels == 2 ? n1 : n1 + n2);
    const uint32_t base = atomicAdd(&a.ctrl[kNParts], np + extra);
    if (np <= a.small_parts) {
        a.small[atomicAdd(&a.ctrl[kNSmall], 1u)] = make_uint4(base, np, bucket, 0u);
        return base;
    }
    uint32_t src = base, cnt = np;
#pragma unroll
    for (int lv = 0; lv < 3; ++lv) {   // the last level has one output
        const uint32_t nout = lv == 2 || lv + 1 == a.levels ? 1u : (cnt + kTreeParts - 1) / kTreeParts;
        const uint32_t e = atomicAdd(&a.ctrl[kNTree + lv], nout);
        if (nout == 1) {
            a.tree[lv][e] = make_uint4(src, cnt, bucket, 0u);
            break;
        }
        for (uint32_t i = 0; i < nout; ++i) {
            const uint32_t left = cnt - i * kTreeParts;
            a.tree[lv][e + i] = make_uint4(src + i * kTreeParts, left < kTreeParts ? left : kTreeParts,
                                           (src + cnt + i) | kPart, 0u);
        }
        src += cnt;
        cnt = nout;
    }
    return base;
}

// A bin of more than kWide pieces, written by its whole block.
constexpr uint32_t kWide = 16;
struct WideBin {
    uint32_t s, np, q, big, dest, at_big, at_q;
};

// The pieces of every bin to their places in the list (longest first) and the merge
// lists; empty buckets get coordinate 2 = 0, which every reader of buckets takes as
// "no point".
__global__ void __launch_bounds__(kPieceThreads) k_piece_emit(PieceArgs a) {
    __shared__ uint32_t h[kMaxPiece + 1], base[kMaxPiece + 1];
    __shared__ uint32_t warp_tot[kPieceThreads / 32];
    __shared__ WideBin wide[kPieceThreads];
    __shared__ uint32_t nwide;
    const int t = threadIdx.x;
    for (uint32_t k = t; k <= kMaxPiece; k += kPieceThreads) h[k] = 0;
    if (t == 0) nwide = 0;
    __syncthreads();
    const size_t id = blockIdx.x * (size_t)kPieceThreads + t;
    const BinRun r = bin_run(a, id);
    uint32_t np = 0, q = 0, big = 0, rank_big = 0, rank_q = 0;
    if (r.m) {
        const uint32_t cap = piece_cap(a);
        np = (r.m + cap - 1) / cap;
        q = r.m / np;
        big = r.m - q * np;
        if (big) rank_big = atomicAdd(&h[q + 1], big);
        rank_q = atomicAdd(&h[q], np - big);
    } else if (r.bucket != kNone) {
        uint4* z = a.buckets + (size_t)r.bucket * kXyzzVec + 6;
        z[0] = z[1] = z[2] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    // Class offsets: lengths in descending order. Thread t has length kMaxPiece - t.
    {
        const uint32_t len = kMaxPiece - t;   // 256 .. 1
        const uint32_t v = len <= a.cap ? a.ctrl[kHist + len] : 0u;
        uint32_t x = v;
        const int lane = t & 31, wid = t >> 5;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[wid] = x;
        __syncthreads();
        uint32_t before = 0;
        for (int k = 0; k < wid; ++k) before += warp_tot[k];
        const uint32_t mine = h[len];
        base[len] = before + x - v + (mine ? atomicAdd(&a.ctrl[kCursor + len], mine) : 0u);
    }
    __syncthreads();
    if (np) {
        uint32_t dest = r.bucket;
        if (np > 1) dest = plan_merge(a, np, r.bucket) | kPart;
        const uint32_t pb = big ? base[q + 1] + rank_big : 0u, pq = base[q] + rank_q;
        if (np <= kWide) {
            uint32_t s = r.s;
            for (uint32_t i = 0; i < np; ++i) {
                const uint32_t len = i < big ? q + 1 : q;
                a.pieces[i < big ? pb + i : pq + i - big] = make_uint4(s, len, dest + i, 0u);
                s += len;
            }
        } else {
            wide[atomicAdd(&nwide, 1u)] = {r.s, np, q, big, dest, pb, pq};
        }
    }
    __syncthreads();
    for (uint32_t k = 0; k < nwide; ++k) {
        const WideBin b = wide[k];
        for (uint32_t i = t; i < b.np; i += kPieceThreads) {
            const bool is_big = i < b.big;
            a.pieces[is_big ? b.at_big + i : b.at_q + i - b.big] =
                make_uint4(b.s + i * b.q + (is_big ? i : b.big), is_big ? b.q + 1 : b.q, b.dest + i, 0u);
        }
    }
}

struct AccArgs {
    const uint32_t* items;   // sorted: stored point | sign << 31
    const uint4* pts;
    uint32_t npts;           // stored points
    uint4* buckets;          // [W][Bp], four coordinates
    uint4* parts;            // partial sums, four coordinates
    const uint4* pieces;
    const uint32_t* hist;    // pieces per length: their sum is the list's length
    uint32_t cap;
};

// Pieces in the list (the same in every thread of the warp).
__device__ __forceinline__ uint32_t piece_count(const AccArgs& a) {
    uint32_t v = 0;
    for (uint32_t k = threadIdx.x & 31; k <= a.cap; k += 32) v += a.hist[k];
    return __reduce_add_sync(0xffffffffu, v);
}

// Sum of one piece to its destination. What bounds it: the integer multiply pipe (7 or
// 10 field products per point); the gather of the next point overlaps the other warps'
// additions.
template <class M>
__device__ __forceinline__ void accumulate_piece(const AccArgs& a, uint32_t id) {
    const uint4 pc = a.pieces[id];
    const uint32_t* it = a.items + pc.x;
    typename M::acc acc;
    uint32_t v = it[0];
    uint32_t idx = v & ~kSign;
    if (idx >= a.npts) idx = 0;   // cannot happen for sorted digit output; keeps reads in bounds
    bool inf = M::first_at(acc, a.pts, idx, (v & kSign) != 0);
    for (uint32_t i = 1; i < pc.y; ++i) {
        v = it[i];
        idx = v & ~kSign;
        if (idx >= a.npts) continue;
        M::madd_at(acc, inf, a.pts, idx, (v & kSign) != 0);
    }
    uint4* d = (pc.z & kPart) ? a.parts + (size_t)(pc.z & ~kPart) * kXyzzVec : a.buckets + (size_t)pc.z * kXyzzVec;
    M::store(d, acc);
}

// Register caps per curve model (M::kAccBlocks blocks of 128 resident per SM), each
// the faster of the caps measured at n = 2^20, c = 16: XYZZ at 168 registers, three
// blocks; Edwards at 128 registers, four blocks.
template <class M>
__global__ void __launch_bounds__(128, M::kAccBlocks) k_accumulate(AccArgs a) {
    const uint32_t n = piece_count(a);
    const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) accumulate_piece<M>(a, id);
}

// Batched MSMs: one persistent kernel drains a queue of the pieces of all jobs. Each
// warp takes 32 consecutive places of one job's list with one atomic; a job's share of
// the queue is its plan's bound on pieces (rounded up to 32), of which only the places
// below its piece count hold work.
constexpr int kMaxBatch = 128;
struct BatchAcc {
    AccArgs job[kMaxBatch];
    uint32_t prefix[kMaxBatch + 1];  // cumulative places over jobs
    int njobs;
    uint32_t* counter;
};

template <class M>
__global__ void __launch_bounds__(128, M::kAccBlocks) k_accumulate_batched(const __grid_constant__ BatchAcc b) {
    const uint32_t total = b.prefix[b.njobs];
    const int lane = threadIdx.x & 31;
    int have = -1;       // the job whose piece count is at hand
    uint32_t count = 0;
    for (;;) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(b.counter, 32u);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= total) break;
        int lo = 0, hi = b.njobs - 1;   // last job with prefix <= base
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (b.prefix[mid] <= base) lo = mid; else hi = mid - 1;
        }
        const AccArgs& a = b.job[lo];
        if (lo != have) {
            count = piece_count(a);
            have = lo;
        }
        const uint32_t id = base - b.prefix[lo] + lane;
        if (id < count) accumulate_piece<M>(a, id);
        __syncwarp();
    }
}

// The block's sum of m points. More than 128 are first summed to 128, one thread each;
// then the block's 32 groups of four lanes sum points g, g + 32, ... in sequence, four
// lanes per addition, and a tree over the groups in shared memory ends it (5 levels).
// Every group of a warp runs the same additions (a missing operand is the identity; idle
// groups of warp 0 add and discard), so each __syncwarp inside them is warp-wide; a warp
// with no active group skips a level as a whole. Thread 0 stores the sum.
constexpr int kTreeThreads = 128;
constexpr int kTreeGroups = kTreeThreads / 4;
constexpr size_t kTreeWave = 152 * 3;  // blocks resident at once (3 per SM)

template <class M>
struct TreeShared {
    uint4 pub[kTreeThreads * kXyzzVec];
    uint4 idn[kXyzzVec];
    fe sh[kTreeGroups][4];
};

template <class M>
__device__ __forceinline__ void tree_init(TreeShared<M>& s) {
    if (threadIdx.x == 0) {
        typename M::acc e;
        M::set_inf(e);
        M::store(s.idn, e);
    }
    __syncthreads();
}

// src(i): the address of point i, or of the identity s.idn.
template <class M, class Src>
__device__ __forceinline__ void block_sum_of(TreeShared<M>& s, const Src& src, uint32_t m, uint4* __restrict__ out) {
    const int t = threadIdx.x, g = t >> 2, l = t & 3, warp = t >> 5;
    typename M::acc acc;
    if (m > kTreeThreads) {   // first by threads, a point of every 128 each
        M::load(acc, src(t));
        for (uint32_t i = t + kTreeThreads; i < m; i += kTreeThreads) M::add_mem(acc, src(i));
        M::store(s.pub + t * kXyzzVec, acc);
        __syncthreads();
        m = kTreeThreads;
        M::load(acc, s.pub + g * kXyzzVec);
        for (uint32_t i = kTreeGroups + g; i < kTreeThreads; i += kTreeGroups)
            M::add4_mem(acc, s.pub + i * kXyzzVec, s.sh[g], l);
        __syncthreads();      // the points are read before the levels below publish over them
    } else {
        M::load(acc, (uint32_t)g < m ? src(g) : s.idn);
        for (uint32_t i0 = kTreeGroups; i0 < m; i0 += kTreeGroups) {
            const uint32_t i = i0 + g;
            M::add4_mem(acc, i < m ? src(i) : s.idn, s.sh[g], l);
        }
    }
    // level h: groups [h, 2h) publish, groups [0, h) add them. The slots read at
    // level h, [h, 2h), are never written at a later level (those write [h', 2h')
    // with 2h' <= h), so one barrier per level orders every access.
    for (int h = kTreeGroups / 2; h >= 1; h >>= 1) {
        if ((uint32_t)h >= m) continue;   // only identities there (block-uniform)
        if (g >= h && g < 2 * h && l == 0) M::store(s.pub + g * kXyzzVec, acc);
        __syncthreads();
        if (warp * 8 < h) {
            typename M::acc r = acc;
            M::add4_mem(r, s.pub + (g + h) * kXyzzVec, s.sh[g], l);  // g + h < 32: g < h for h >= 8, g <= 7 below
            if (g < h) acc = r;
        }
    }
    if (t == 0) M::store(out, acc);
}

template <class M>
__device__ __forceinline__ void block_sum(TreeShared<M>& s, const uint4* __restrict__ in, uint32_t m, uint4* __restrict__ out) {
    block_sum_of(s, [&](uint32_t i) { return in + (size_t)i * kXyzzVec; }, m, out);
}

__device__ __forceinline__ uint4* merge_dest(uint4* parts, uint4* buckets, uint32_t d) {
    return (d & kPart) ? parts + (size_t)(d & ~kPart) * kXyzzVec : buckets + (size_t)d * kXyzzVec;
}

// One level of the merge: the tree entries by blocks, then (nsmall not null) the buckets
// of few parts by threads.
template <class M>
__global__ void __launch_bounds__(kTreeThreads) k_merge_parts(uint4* parts, uint4* buckets, const uint4* __restrict__ tree,
                                                              const uint32_t* __restrict__ ntree,
                                                              const uint4* __restrict__ small,
                                                              const uint32_t* __restrict__ nsmall) {
    __shared__ TreeShared<M> s;
    const uint32_t nt = *ntree;
    if (blockIdx.x < nt) {
        tree_init(s);
        for (uint32_t e = blockIdx.x; e < nt; e += gridDim.x) {
            const uint4 x = tree[e];
            block_sum(s, parts + (size_t)x.x * kXyzzVec, x.y, merge_dest(parts, buckets, x.z));
            __syncthreads();   // the published points are read before the next entry's
        }
    }
    if (!nsmall) return;
    const uint32_t ns = *nsmall;
    // from the last block down: the first ones have the tree entries
    for (uint32_t i = (gridDim.x - 1 - blockIdx.x) * kTreeThreads + threadIdx.x; i < ns; i += gridDim.x * kTreeThreads) {
        const uint4 x = small[i];
        const uint4* p = parts + (size_t)x.x * kXyzzVec;
        typename M::acc acc;
        M::load(acc, p);
        for (uint32_t k = 1; k < x.y; ++k) M::add_mem(acc, p + (size_t)k * kXyzzVec);
        M::store(buckets + (size_t)x.z * kXyzzVec, acc);
    }
}

// ---------------------------------------------------------------- stage 6

// Thread (wi, g): Y = sum_{i=1..L} B[gL+i], V = sum_{i=1..L} i * B[gL+i] (bucket b at
// index b-1): 2 (L - 1) additions.
template <class M>
__global__ void __launch_bounds__(128) k_reduce_segments(const uint4* __restrict__ buckets, uint32_t Bp, uint32_t L, int w0, int nwin,
                                  uint32_t G, uint4* __restrict__ Y, uint4* __restrict__ V) {
    const size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (id >= (size_t)nwin * G) return;
    const size_t wi = id / G, g = id % G;
    const uint4* seg = buckets + ((size_t)(w0 + wi) * Bp + g * L) * kXyzzVec;
    typename M::acc T, S;
    const uint4* last = seg + (size_t)(L - 1) * kXyzzVec;
    if (M::empty(last))
        M::set_inf(T);
    else
        M::load(T, last);
    S = T;
    for (int i = (int)L - 1; i >= 1; --i) {
        M::add_mem(T, seg + (size_t)(i - 1) * kXyzzVec);   // T += B
        M::add(S, T);                                       // S += T
    }
    M::store(Y + id * kXyzzVec, T);
    M::store(V + id * kXyzzVec, S);
}

__device__ __forceinline__ void shfl_xor_words(fe& r, const fe& a) {
#pragma unroll
    for (int k = 0; k < fq::N; ++k) r.v[k] = __shfl_xor_sync(0xffffffffu, a.v[k], 1);
}

__device__ __forceinline__ void ModelXyzz::exchange(acc& Q, const acc& P) {
    shfl_xor_words(Q.X, P.X);
    shfl_xor_words(Q.Y, P.Y);
    shfl_xor_words(Q.ZZ, P.ZZ);
    shfl_xor_words(Q.ZZZ, P.ZZZ);
}
__device__ __forceinline__ void ModelEdwards::exchange(acc& Q, const acc& P) {
    shfl_xor_words(Q.X, P.X);
    shfl_xor_words(Q.Y, P.Y);
    shfl_xor_words(Q.Z, P.Z);
    shfl_xor_words(Q.T, P.T);
}

// The same sums by two lanes per segment: the even lane runs T, the odd lane S one step
// behind it, so a segment takes L additions in sequence instead of 2 (L - 1), and as many
// threads serve half as many segments of twice the length: the bit sums that follow have
// half the points. Measured, with the bit sums: 2^18 Edwards buckets 192 + 160 -> 222 + 106 us,
// 17 windows of 2^14 XYZZ buckets 273 + 282 -> 307 + 175 us. At 2^19 XYZZ buckets the multiply
// pipe bounds the one-thread form (580 us) and the estimate keeps it.
template <class M>
__global__ void __launch_bounds__(128) k_reduce_pairs(const uint4* __restrict__ buckets, uint32_t Bp, uint32_t L, int w0, int nwin,
                               uint32_t G, uint4* __restrict__ Y, uint4* __restrict__ V) {
    const size_t nseg = (size_t)nwin * G;
    size_t id = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 1;
    const bool run_s = threadIdx.x & 1, live = id < nseg;
    if (!live) id = nseg - 1;   // whole warps go through the exchanges
    const size_t wi = id / G, g = id % G;
    const uint4* seg = buckets + ((size_t)(w0 + wi) * Bp + g * L) * kXyzzVec;
    typename M::acc P, Q;
    M::set_inf(P);
    if (!run_s && !M::empty(seg + (size_t)(L - 1) * kXyzzVec)) M::load(P, seg + (size_t)(L - 1) * kXyzzVec);
#pragma unroll 1
    for (uint32_t i = 1; i <= L; ++i) {
        M::exchange(Q, P);      // the odd lane adds T as it stands
        if (!run_s) {           // the even lane the next bucket
            M::set_inf(Q);
            if (i < L) {
                const uint4* b = seg + (size_t)(L - 1 - i) * kXyzzVec;
                if (!M::empty(b)) M::load(Q, b);
            }
        }
        M::add(P, Q);
    }
    if (live) M::store((run_s ? V : Y) + id * kXyzzVec, P);
}

// Sums of the segments' points by the bits of their index, four lanes per addition.
// Per window there are (logG + 2) nb blocks: block (k, q), k < logG, sums the q-th of nb
// equal slices of the G/2 points Y_g with bit k of g set (the j-th such index is j with
// a one inserted at bit k); the last 2 nb blocks sum slices of all V_g. Every block
// sums (G/2) / nb points (block_sum_of). What bounds it is the latency of its additions:
// 5.7 (Edwards) or 11 us (XYZZ) each on four lanes while the blocks fit two per SM, about
// twice that on one thread. One thread per slice of eight points and a launch of block
// trees over the slices took 87 + 29 us where this takes 51 + 8 (Edwards, 13 windows of 512
// buckets) and 145 + 68 us where this takes 78 (XYZZ, 32 windows of 256). kRaw:
// Y = V are the buckets themselves (L = 1), which may be empty.
template <class M, bool kRaw>
__global__ void __launch_bounds__(kTreeThreads) k_bit_sums(const uint4* __restrict__ Y, const uint4* __restrict__ V, int nwin,
                                                          uint32_t G, int logG, uint32_t nb, uint4* __restrict__ P) {
    __shared__ TreeShared<M> s;
    const uint32_t per_w = (uint32_t)(logG + 2) * nb;
    const uint32_t wi = blockIdx.x / per_w, r = blockIdx.x % per_w;
    if (wi >= (uint32_t)nwin) return;  // whole block
    tree_init(s);
    const uint32_t k = r / nb;
    auto at_point = [&](const uint4* q) { return kRaw && M::empty(q) ? (const uint4*)s.idn : q; };
    if (k < (uint32_t)logG) {
        const uint32_t span = (G / 2) / nb, j0 = (r % nb) * span, low = (1u << k) - 1u;
        const uint4* y = Y + (size_t)wi * G * kXyzzVec;
        block_sum_of(s, [&](uint32_t i) {
            const uint32_t j = j0 + i, g = ((j & ~low) << 1) | (1u << k) | (j & low);
            return at_point(y + (size_t)g * kXyzzVec);
        }, span, P + (size_t)blockIdx.x * kXyzzVec);
    } else {
        const uint32_t v = r - (uint32_t)logG * nb;                     // slice of 2 nb
        const uint32_t g0 = (uint32_t)((uint64_t)v * G / (2 * nb)), g1 = (uint32_t)((uint64_t)(v + 1) * G / (2 * nb));
        const uint4* x = V + ((size_t)wi * G + g0) * kXyzzVec;
        block_sum_of(s, [&](uint32_t i) { return at_point(x + (size_t)i * kXyzzVec); }, g1 - g0,
                     P + (size_t)blockIdx.x * kXyzzVec);
    }
}

// Block seg: out[seg] = the sum of in[seg][0 .. m - 1].
template <class M>
__global__ void __launch_bounds__(kTreeThreads) k_sum_rows(const uint4* __restrict__ in, uint32_t m, uint4* __restrict__ out) {
    __shared__ TreeShared<M> s;
    tree_init(s);
    block_sum(s, in + (size_t)blockIdx.x * m * kXyzzVec, m, out + (size_t)blockIdx.x * kXyzzVec);
}

// ---------------------------------------------------------------- stage 7

// The two latency-bound chains run on one group of four warps per block: each point
// operation's products are spread over the warps (one product per warp and formula
// level) and each product over the lanes of its warp (wred.cuh). The next operand's
// loads are issued before the current operation, so they overlap it.

// Block w: S_w = L sum_{k < logG} 2^k Z_k + Z_logG + Z_(logG + 1) for window w (the last
// two: the halves of sum_g V_g), by Horner from the top term; S_w is left in the chain's operand form (limbs).
template <class M>
__global__ void __launch_bounds__(128, 1) k_window_horner_w(const uint4* __restrict__ Z, int nwin, int logG, int log2L,
                                                         int* __restrict__ S) {
    using C = typename M::chain;
    __shared__ __align__(16) int mem[wred::kSharedWords];
    const int w = blockIdx.x;
    if (w >= nwin) return;  // whole block
    wred::Group g;
    wred::init(g, mem);
    C::load_const(g);
    const uint32_t* z = reinterpret_cast<const uint32_t*>(Z + (size_t)w * (logG + 2) * kXyzzVec);
    constexpr size_t kWords = 4 * kXyzzVec;
    C::set_inf(g);
    wred::Packed next = wred::load_packed(g, z + (size_t)(logG > 0 ? logG - 1 : logG) * kWords);
    for (int k = logG - 1; k >= 0; --k) {
        const wred::Packed q = next;   // Z_k
        next = wred::load_packed(g, z + (size_t)(k > 0 ? k - 1 : logG) * kWords);
        if (k < logG - 1) C::dbl(g, true);
        C::set_operand(g, q.limb, wred::zero_z(g, q));
        C::add(g);
    }
    for (int t = 0; t < log2L; ++t) C::dbl(g, t == log2L - 1);
    for (int h = 0; h < 2; ++h) {
        const wred::Packed q = next;   // Z_(logG + h)
        if (h == 0) next = wred::load_packed(g, z + (size_t)(logG + 1) * kWords);
        C::set_operand(g, q.limb, wred::zero_z(g, q));
        C::add(g);
    }
    const int v = C::as_operand(g);
    if (g.lane < 16) S[(size_t)w * wred::kLimbPointWords + 16 * g.w + g.lane] = v;
}

// sum_w 2^(c w) S_w by Horner over the windows, then the affine result in standard
// form.
template <class M>
__global__ void __launch_bounds__(128, 1) k_chain_w(const int* __restrict__ S, int W, int c, uint32_t* __restrict__ out) {
    using C = typename M::chain;
    __shared__ __align__(16) int mem[wred::kSharedWords];
    wred::Group g;
    wred::init(g, mem);
    C::set_inf(g);
    int next = wred::load_limbs(g, S + (size_t)(W - 1) * wred::kLimbPointWords);
    for (int j = W - 1; j >= 0; --j) {
        g.st(wred::kQ + g.w, next);    // S_j (the operand slots are read before an addition's last barrier)
        if (j > 0) next = wred::load_limbs(g, S + (size_t)(j - 1) * wred::kLimbPointWords);
        if (j < W - 1)
            for (int t = 0; t < c; ++t) C::dbl(g, t == c - 1);
        else
            __syncthreads();
        C::add(g);
    }
    C::store_affine(g, out);
}

// ---------------------------------------------------------------- planning

struct Plan {
    size_t n;        // scalars (and input points)
    size_t np;       // stored points = items per window: n, or 2n with GLV
    int edw, glv;    // curve model (0 XYZZ, 1 Edwards); GLV split
    int pre;         // precomputed shifted points: the Wd digit windows share one bucket set
    int Wd;          // digit windows per scalar (W = 1 when pre, else W = Wd)
    size_t items;    // items per pipeline window: np, or Wd np when pre
    int stored_vec;  // uint4 per stored point
    int user_bits;   // scalar range checked against opts.scalar_bits
    int c, sgn, bits, W;
    uint32_t B, Bp;
    int passes, rb;  // radix-sort passes of rb-bit digits
    size_t tiles;
    int K;          // longest piece of a bucket's run
    int K_few;      // and where few digits are nonzero, at least (piece_cap)
    size_t shared;  // half a thread's share of the batch (0: a single call)
    int levels;     // tree levels of the merge
    size_t wave;    // resident accumulation threads
    uint32_t small_parts;   // parts that one thread puts together
    size_t max_pieces, max_parts, max_small, max_tree[3];   // per group: bounds over any digits
    int gw;         // windows per group
    int ngroups;
    uint32_t L, G;
    uint32_t nb;     // blocks per bit of the segment sums
    bool pairs;      // segments by two lanes each
    int logG, log2L;
    size_t off_status, off_ctrl, ctrl_bytes;   // status words, then the groups' counters: cleared together
    size_t off_points, off_keys0, off_vals0, off_keys1, off_vals1, off_rank, off_hist, off_dtot;
    int counting;                      // counting sort (else LSD radix sort)
    size_t nbins, off_bins, off_bsum;  // counting sort: bins (window, key) and scan tile totals
    uint32_t ttiles, tT;               // counting sort in shared-memory tiles: tiles per window, items per
                                       // tile (ttiles = 0: global counters)
    size_t off_tcnt;                   // per-tile counts and prefixes [W][ttiles][Bp + 1]
    size_t off_buckets, off_parts, off_pieces, off_small, off_tree[3], off_Y, off_V, off_P0, off_P1;
    size_t off_S, total;
};


int ilog2(uint64_t v) {
    int r = 0;
    while ((1ull << (r + 1)) <= v) ++r;
    return r;
}

// Tuned schedules for signed digits by floor(log2 n), one table per mode (Edwards,
// GLV, fixed-base), set from measured tables by msm_g1_set_window_table (window
// widths) and msm_g1_set_schedule (every field); 0 = the built-in rule.
std::atomic<int> g_ctable[8][32];      // window width c
std::atomic<int> g_ktable[8][32];      // longest piece K
std::atomic<int> g_sorttable[8][32];   // 1 counting sort, 2 LSD radix sort
std::atomic<int> g_rtable[8][32];      // log2 of the level-1 reduction threads
std::atomic<int> g_gtable[8][32];      // window groups (1 = no overlap of tails with accumulation)

int table_mode(uint32_t flags) {
    return ((flags & MSM377_EDWARDS) ? 1 : 0) | ((flags & MSM377_GLV) ? 2 : 0) |
           ((flags & MSM377_PRECOMPUTED) ? 4 : 0);
}

// Window width by floor(log2 n) for signed digits, per mode (bit 0 Edwards, bit 1 GLV):
// the fastest of the widths 4..17 on GB300 at 1.05 and 1.55 times each power of two (the
// better of the two on average). A wider window means fewer windows but more buckets; which
// widths pay also depends on the top window, which is short (and its few buckets heavy) when
// c just fails to divide the scalar's bits: with GLV's 127-bit halves 11 and 16 divide well, so
// with Edwards + GLV 2^12 .. 2^14 takes 11 and 2^17 .. 2^22 16 (n = 2.7 * 10^5: c = 14 1965, 15 1721,
// 16 1596, 17 1869 us). That sweep came before the merged Y3 of XYZZ additions, the two-lane
// segment sums and the shorter pieces; measured again with them (widths 3..18, 2^4 .. 2^22), the
// entries are within 2.1 % of the fastest width but for these: c = 8 at 2^4 and 2^5 is 2 to
// 9 % faster in every mode; XYZZ 2^12: 11 5.5 %, 2^16: 14 3.6 %; GLV 2^20: 16 3.6 %, 2^21 and 2^22:
// 18 2.7 and 5.0 %.
constexpr int kDefaultLogs = 23;
constexpr int8_t kDefaultC[4][kDefaultLogs] = {
    {4, 4, 4, 4, 4, 4, 6, 6, 7, 7, 8, 11, 8, 11, 11, 13, 13, 15, 15, 16, 16, 17, 17},   // XYZZ
    {4, 4, 4, 4, 4, 4, 5, 5, 6, 7, 8, 8, 11, 11, 11, 11, 14, 15, 15, 16, 16, 17, 17},   // Edwards
    {4, 4, 4, 4, 4, 4, 4, 4, 4, 4, 9, 10, 11, 11, 11, 14, 15, 16, 16, 16, 17, 17, 17},  // XYZZ + GLV
    {4, 4, 4, 4, 4, 4, 4, 4, 5, 5, 5, 8, 11, 11, 11, 12, 15, 16, 16, 16, 16, 16, 16}};  // Edwards + GLV

// single: one call on its own, whose latency counts. The jobs of a batch overlap, so their
// total work counts, and there the rule by size below is the better one (24 jobs of 2^10
// to 2^18 points: 7.25 ms, 7.33 with the table). Installed widths are measured on single calls
// too and are not taken there either (30 jobs of 2^10 to 2^13 points, Edwards + GLV, in one
// graph: 1964 us by the rule, 2354 with a tuned table; 24 of 2^10 to 2^18 8748 and 8930).
int default_c(size_t n, int sgn, uint32_t flags, bool single = true) {
    int lg = n > 1 ? ilog2(n) : 0;
    if (single && sgn && lg < 32) {
        const int t = g_ctable[table_mode(flags)][lg].load(std::memory_order_relaxed);
        if (t > 0) return t;
    }
    if (single && sgn && !(flags & MSM377_PRECOMPUTED))
        return kDefaultC[table_mode(flags) & 3][lg < kDefaultLogs ? lg : kDefaultLogs - 1];
    if (flags & MSM377_GLV) ++lg;  // 2n points per window
    if (flags & MSM377_PRECOMPUTED) lg += 2;  // one bucket set for all windows: wider windows pay
    int c = lg - 4;
    if (!sgn) c = lg - 3;
    if (c < 4) c = 4;
    if (c > 17) c = 17;
    return c;
}

constexpr int kMaxGroups = 8;

// single = false (batched calls): one window group; whole jobs overlap instead.
// batch_items: items of all jobs of the batch.
bool make_plan(size_t n, const msm_opts* o, Plan* p, bool single = true, size_t batch_items = 0) {
    if (!o) return false;
    p->n = n;
    p->edw = (o->flags & MSM377_EDWARDS) ? 1 : 0;
    p->glv = (o->flags & MSM377_GLV) ? 1 : 0;
    p->pre = (o->flags & MSM377_PRECOMPUTED) ? 1 : 0;
    // precomputed sets are Edwards stored points made for one explicit c
    if (p->pre && (!p->edw || !(o->flags & MSM377_POINTS_PREPARED) || o->c == 0)) return false;
    p->stored_vec = p->edw ? ModelEdwards::kStored : ModelXyzz::kStored;
    p->sgn = o->signed_digits ? 1 : 0;
    p->user_bits = o->scalar_bits ? o->scalar_bits : 256;
    if (p->user_bits < 1 || p->user_bits > 256) return false;
    p->bits = p->glv ? 127 : p->user_bits;  // GLV halves are below 2^127
    p->c = o->c ? o->c : default_c(n, p->sgn, o->flags, single);
    if (p->c < 2 || p->c > 20) return false;
    if (n >= (1ull << 30)) return false;
    const size_t np = p->glv ? 2 * n : n;
    p->np = np;
    p->Wd = p->sgn ? (p->bits + 1 + p->c - 1) / p->c : (p->bits + p->c - 1) / p->c;
    p->W = p->pre ? 1 : p->Wd;
    p->items = p->pre ? (size_t)p->Wd * np : np;
    if (p->items >= (1ull << 31)) return false;
    if ((uint64_t)p->W * p->items >= (1ull << 32)) return false;   // bin offsets are 32-bit
    const size_t items = p->items;
    p->B = p->sgn ? (1u << (p->c - 1)) : ((1u << p->c) - 1u);
    p->Bp = p->sgn ? p->B : (1u << p->c);
    // keys are |digit| <= 2^(c-1) (signed) or < 2^c: c bits, sorted 8 bits per pass
    // (10-bit digits would save a pass at c = 17..20 but measured slower on GB300:
    // the 1024-bin scatter's shared-memory counters cost more than the pass)
    p->rb = 8;
    p->passes = (p->c + p->rb - 1) / p->rb;
    // Measured on GB300: the counting sort (ranks taken in the counting pass, no
    // atomics in the scatter) beats the radix passes for every plan; the radix sort
    // stays available for comparison.
    const int lgn = n > 1 ? ilog2(n) : 0;
    const int tmode = table_mode(o->flags);
    // installed entries measured on single calls rule these only (default_c); the sort is a
    // choice for any call
    const int tsort = (p->sgn && lgn < 32) ? g_sorttable[tmode][lgn].load(std::memory_order_relaxed) : 0;
    const int tk = (single && p->sgn && lgn < 32) ? g_ktable[tmode][lgn].load(std::memory_order_relaxed) : 0;
    const int tr = (single && p->sgn && lgn < 32) ? g_rtable[tmode][lgn].load(std::memory_order_relaxed) : 0;
    const int tg = (p->sgn && lgn < 32) ? g_gtable[tmode][lgn].load(std::memory_order_relaxed) : 0;
    p->counting = ((o->flags & MSM377_RADIX_SORT) || tsort == 2) ? 0 : 1;
    p->tiles = (items + kSortTile - 1) / kSortTile;
    // Counting in shared-memory tiles when a block's packed counters fit: tiles of
    // fewer than 2^16 items, about one wave of 1024-thread blocks (two per SM when
    // the counters take at most 100 KB), and at least ~1024 items a tile.
    p->ttiles = 0;
    p->tT = 0;
    {
        const size_t smem = (size_t)((p->Bp + 2) / 2) * 4;
        if (p->counting && items > 0 && smem <= kTileSmemMax) {
            const size_t per_sm = smem <= 100 * 1024 ? 2 : 1;
            const size_t fewest = (items + kTileItemsMax - 1) / kTileItemsMax;
            size_t tl = (152 * per_sm + p->W - 1) / p->W;
            const size_t cap = (items + 1023) / 1024;
            if (tl > cap) tl = cap;
            if (tl < fewest) tl = fewest;
            if (tl < 1) tl = 1;
            p->ttiles = (uint32_t)tl;
            p->tT = (uint32_t)((items + tl - 1) / tl);
        }
    }
    // Window groups (a schedule option): the accumulation runs group by group on the
    // caller's stream and each group's merges, bucket reduction and per-window sums
    // run on a higher-priority helper stream as soon as its accumulation is done,
    // overlapping the next group's accumulation. Built-in rule: one group. Measured
    // on GB300 (Edwards + GLV, c = 16): 2^20 one group 6.17 ms, two 6.55, four 7.28;
    // 2^22 20.7 / 22.0 / 22.6 ms -- the overlapped tails slow the accumulation more
    // than they save, so the autotuner keeps one group at every size measured.
    int groups = 1;
    if (single && !p->pre) {
        groups = tg > 0 ? tg : 1;
        if (groups > p->W) groups = p->W;
        if (groups > kMaxGroups) groups = kMaxGroups;
    }
    p->gw = (p->W + groups - 1) / groups;
    p->ngroups = (p->W + p->gw - 1) / p->gw;
    // Pieces of at most K items, one thread each (stage 4): K = the mean run plus four
    // standard deviations, so that with at least a wave of buckets only unusually long
    // runs are cut (random digits leave hardly any); up to a third of a resident thread's
    // share of all items, so that a piece never outlasts the rest of the work, and up
    // to one or two shares, so that every resident thread (152 SMs x kAccBlocks blocks of 128 on
    // a GB300) has work where buckets are few.
    const size_t kWave = (size_t)152 * 128 * (p->edw ? ModelEdwards::kAccBlocks : ModelXyzz::kAccBlocks);
    const size_t total = (size_t)p->gw * items;
    const size_t mean = (items + p->B - 1) / p->B;      // items per bucket of a full window
    size_t K = mean + 8;
    while ((K - mean) * (K - mean) < 16 * mean) ++K;    // mean + 4 sqrt(mean)
    const size_t share = (total + kWave - 1) / kWave;
    if (K < share / 3) K = share / 3;
    // In a batch the jobs fill the threads together: pieces may be as long as half a
    // thread's share of the whole batch, and fewer sums of parts are left to merge; but no
    // longer than 48 on that account, as the queue's last job would end late (30 jobs of
    // 2^10 to 2^13 points 2.65 -> 2.19 ms; 24 of 2^10 to 2^18 7.17 -> 6.94, without the 48 7.24).
    const size_t shared = batch_items / kWave / 2 < 48 ? batch_items / kWave / 2 : 48;
    // Long shares: little more than one, or runs shorter than expected (zero digits) stay
    // whole and leave threads idle where buckets are fewer than threads; short shares: two,
    // as the parts' merges cost more there. Against two shares throughout, c = 12, XYZZ:
    // 262144 GLV pairs, half the digits zero, 2819 -> 1845 us; 262144 points 3411 -> 2720 us. One
    // share throughout: 30071 GLV pairs, c = 9, 960 -> 1426 us.
    const size_t two = 2 * share + 4, most = batch_items ? two : std::max(share + 4, std::min<size_t>(two, 36));
    const size_t longest = most > shared ? most : shared;
    // where few digits are nonzero: no shorter than the merges are worth, nor, in a batch, than
    // for the job alone
    const size_t few = batch_items ? two : 36;
    if (K > longest) K = longest;
    if (K < 2) K = 2;
    if (K > kMaxPiece) K = kMaxPiece;
    if (tk > 0) K = (size_t)tk;        // measured choice (2..256)
    p->K = (int)K;
    p->K_few = tk > 0 || K < few ? (int)K : (int)few;
    p->shared = batch_items / kWave / 2;
    p->wave = kWave;
    {
        const size_t parts = (items + K - 1) / K;   // of one bucket, all digits nonzero
        p->levels = parts > (size_t)kTreeParts * kTreeParts ? 3 : parts > kTreeParts ? 2 : items > (size_t)p->K_few ? 1 : 0;
    }
    {
        // sum over buckets of ceil(m / K): at most one piece more than m / K per bucket in
        // use; a bucket with parts has more than K items
        const size_t nbk = (size_t)p->gw * p->Bp, used = nbk < total ? nbk : total;
        const size_t cut = total / (K + 1) < nbk ? total / (K + 1) : nbk;
        p->max_pieces = total / K + used;
        const size_t multi = total / K + cut;
        p->max_parts = multi + multi / 2;               // and the tree levels' sums
        p->max_small = cut;
        // With many buckets the threads' sequential sums fill the GPU; few buckets' parts
        // go to blocks (816 buckets of 8 parts, XYZZ: 195 us by blocks, 280 us by threads).
        p->small_parts = nbk >= 2048 ? 8 : 2;
        // An installed K may cut most buckets into more parts than that: then the longest
        // buckets' additions in sequence on one thread, half as many again as the mean's, against
        // a block for every kTreeParts parts of a bucket (times of one addition as in the bucket
        // reduction below). K = 2, n = 2^20, c = 16: XYZZ 102.2 -> 17.0, Edwards + GLV
        // 21.0 -> 8.7 ms.
        const size_t parts = (mean + K - 1) / K;
        if (tk > 0 && nbk >= 2048 && parts >= p->small_parts) {
            const double full = (double)nbk / (double)kWave;
            const double t1 = p->edw ? std::max(10.5, 25.0 * full) : std::max(18.0, 29.0 * full);
            const size_t of_block = std::min<size_t>(parts, kTreeParts);
            const size_t blocks = nbk * ((parts + kTreeParts - 1) / kTreeParts), steps = (of_block + kTreeGroups - 1) / kTreeGroups + 4;
            const double t4 = (p->edw ? 7.5 : 24.0) * (double)blocks / (double)kTreeWave;
            if (1.5 * (double)parts * t1 < (double)steps * t4) p->small_parts = (uint32_t)(2 * parts);
        }
        // a bucket of more than small_parts parts has an entry for each kTreeParts of them: at
        // most a 32nd of its parts, or one
        p->max_tree[0] = multi / std::min<size_t>(p->small_parts + 1, kTreeParts / 2) + 1;
        p->max_tree[1] = p->max_tree[2] = multi / kTreeParts + 1;
        if (p->max_parts >= kPart || p->max_pieces >= (1ull << 32)) return false;
    }
    // Bucket reduction: segments of L buckets summed by a thread each (2 (L - 1)
    // additions in sequence), then blocks of four-lane additions over the W G segment
    // sums (k_bit_sums). L is the power of two with the least estimated time, from the
    // measured time of one addition alone and of one per resident thread with the GPU
    // full: 10.5 and 25 us on one thread (Edwards; XYZZ 18 and 29 us), 5.7 and 7.5 us (11 and
    // 24 us) on four lanes with three blocks per SM. Small calls take L = 1 or 2, 2^19 buckets L = 16.
    {
        const double t1 = p->edw ? 10.5 : 18.0, t1_full = p->edw ? 25.0 : 29.0;
        const double t4 = p->edw ? 5.7 : 11.0, t4_full = p->edw ? 7.5 : 24.0;
        double best = 0;
        p->L = 0;
        for (uint32_t L = 1; L <= p->Bp; L <<= 1) {
            const uint32_t G = p->Bp / L;
            const int lg = ilog2(G);
            const size_t per_nb = (size_t)p->gw * (lg + 2);
            const double threads = (double)p->gw * G / (double)kWave;
            const double add1 = t1 > t1_full * threads ? t1 : t1_full * threads;
            const double add2 = 1.1 * (t1 > 2 * t1_full * threads ? t1 : 2 * t1_full * threads);
            const bool pairs = L >= 4 && L * add2 < 2.0 * (L - 1) * add1;
            const double segments = L == 1 ? 0.0 : 3.0 + (pairs ? L * add2 : 2.0 * (L - 1) * add1);
            // a tuned number of segments: the longest L that leaves as many
            const bool forced = tr > 0;
            if (forced && L > 1 && (uint64_t)p->W * G < (1ull << tr)) break;
            if (forced) p->L = 0;
            for (uint32_t nb = 1; nb == 1 || (per_nb * nb <= kTreeWave && G / 2 / nb >= (uint32_t)kTreeGroups); nb <<= 1) {
                const double blocks = (double)(per_nb * nb) / (double)kTreeWave;
                const double in_blocks = blocks * kTreeWave * kTreeThreads / (double)kWave;
                const uint32_t span = G / 2 / nb, by_thread = span > kTreeThreads ? span / kTreeThreads - 1 : 0;
                const double steps = (double)((span < kTreeThreads ? span : kTreeThreads) + kTreeGroups - 1) / kTreeGroups + 4;
                const double t = segments +
                                 by_thread * (t1 > t1_full * in_blocks ? t1 : t1_full * in_blocks) +
                                 steps * (t4 > t4_full * blocks ? t4 : t4_full * blocks) +
                                 (nb > 1 ? 3.0 + t4 * ilog2(nb) : 0.0);
                if (p->L == 0 || t < best) {
                    best = t;
                    p->L = L;
                    p->nb = nb;
                    p->pairs = pairs;
                }
            }
        }
    }
    p->G = p->Bp / p->L;
    p->logG = ilog2(p->G);
    p->log2L = ilog2(p->L);
    // workspace layout, 256-byte aligned pieces
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o2 = off;
        off = msm377::align_up(off + bytes, 256);
        return o2;
    };
    const size_t XY = kXyzzBytes;
    p->off_status = take(256);
    p->off_ctrl = take((size_t)p->ngroups * kCtrlWords * 4);
    p->ctrl_bytes = p->off_ctrl + (size_t)p->ngroups * kCtrlWords * 4 - p->off_status;
    p->off_points = take(o->flags & MSM377_POINTS_PREPARED ? 0 : np * 16 * (size_t)p->stored_vec);
    const size_t all = (size_t)p->W * items;
    p->off_keys0 = take(all * 4);
    p->off_vals0 = take(all * 4);
    // the radix sort's ping-pong buffers
    p->off_keys1 = take(p->counting ? 0 : all * 4);
    p->off_vals1 = take(p->counting ? 0 : all * 4);
    p->off_rank = take(p->counting ? all * 4 : 0);  // counting sort: rank within the bin
    p->off_hist = take((size_t)p->W * (1u << p->rb) * (p->tiles ? p->tiles : 1) * 4);
    p->off_dtot = take((size_t)p->W * (1u << p->rb) * 4);
    p->nbins = (size_t)p->W * (p->Bp + 1);  // keys 0 .. Bp of every window
    p->off_bins = take(p->nbins * 4);
    p->off_bsum = take(((p->nbins + kBinBlock - 1) / kBinBlock) * 4);
    p->off_tcnt = take((size_t)p->W * p->ttiles * (p->Bp + 1) * 4);
    p->off_buckets = take((size_t)p->W * p->Bp * XY);
    p->off_parts = take(p->ngroups * p->max_parts * XY);
    p->off_pieces = take(p->ngroups * p->max_pieces * 16);
    p->off_small = take(p->ngroups * p->max_small * 16);
    for (int k = 0; k < 3; ++k) p->off_tree[k] = take(p->ngroups * p->max_tree[k] * 16);
    const size_t segs = p->L > 1 ? (size_t)p->ngroups * p->gw * p->G : 0;   // per group
    p->off_Y = take(segs * XY);
    p->off_V = take(segs * XY);
    const size_t zs = (size_t)p->ngroups * p->gw * (p->logG + 2);
    p->off_P0 = take(zs * p->nb * XY);
    p->off_P1 = take(p->nb > 1 ? zs * XY : 0);
    p->off_S = take((size_t)p->W * wred::kLimbPointWords * sizeof(int));
    p->total = off;
    return true;
}

// Stored points of a set: the form the pipeline gathers from (XYZZ: Montgomery
// affine, 96 B; Edwards: (x, y, k x y), 144 B), for n input points or, with GLV,
// for the 2n points P_0, phi(P_0), P_1, phi(P_1), ...
size_t stored_count(size_t n, uint32_t flags) { return (flags & MSM377_GLV) ? 2 * n : n; }
int stored_vec(uint32_t flags) { return (flags & MSM377_EDWARDS) ? ModelEdwards::kStored : ModelXyzz::kStored; }

// Stored rows of input points [a, b) (rows [a, b), or [2a, 2b) with GLV). The
// Edwards kernel's points per lane are sized for `sizing` points (0: b - a), so the
// launches of the chunks of one set, on separate streams, fill the GPU together.
void launch_prepare_range(const uint4* in, uint4* out, size_t n, size_t a, size_t b, uint32_t flags,
                          cudaStream_t s, size_t sizing = 0) {
    const size_t np = stored_count(n, flags);
    const size_t lo = stored_count(a, flags), hi = stored_count(b, flags);
    if (hi <= lo) return;
    if (flags & MSM377_EDWARDS) {
        // K points per lane: enough batches to give every resident warp (per_sm blocks
        // of 4 warps per SM) about one, at least 2 and at most 32 points per lane
        int dev = 0, sms = 152;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int per_sm = prep_blocks_per_sm((flags & MSM377_GLV) != 0);
        const size_t items = b - a, slots = (size_t)sms * per_sm * 4;
        const size_t basis = sizing ? sizing : items;
        size_t K = (basis + 32 * slots - 1) / (32 * slots);
        K = K < 2 ? 2 : (K > 32 ? 32 : K);
        const size_t batches = (items + 32 * K - 1) / (32 * K);
        const size_t blocks = (batches + 3) / 4;
        const size_t cap = (size_t)sms * per_sm;
        const unsigned grid = (unsigned)(blocks < cap ? blocks : cap);
        if (flags & MSM377_GLV)
            k_prepare_ed<true><<<grid, 128, 0, s>>>(in, out, a, b, (int)K);
        else
            k_prepare_ed<false><<<grid, 128, 0, s>>>(in, out, a, b, (int)K);
    } else {
        k_prepare<<<msm377::grid_for(hi - lo, 256), 256, 0, s>>>(in, out, n, np, lo, hi);
    }
    msm377::note_launches(1);
}

void launch_prepare(const uint4* in, uint4* out, size_t n, uint32_t flags, cudaStream_t s) {
    launch_prepare_range(in, out, n, 0, n, flags, s);
}

template <typename T>
T* at(void* ws, size_t off) {
    return reinterpret_cast<T*>(static_cast<char*>(ws) + off);
}

}  // namespace

using namespace msm377;

extern "C" int msm_g1_default_c(size_t n, int signed_digits, uint32_t flags) {
    return default_c(n, signed_digits ? 1 : 0, flags);
}

extern "C" int msm_g1_set_window_table(const int32_t* c_by_log2n, int len, uint32_t flags) {
    if (len < 0 || len > 32 || (len > 0 && !c_by_log2n))
        return set_error(MSM377_EINVAL, "msm_g1_set_window_table: bad table (len %d)", len);
    if (flags & ~(MSM377_EDWARDS | MSM377_GLV | MSM377_PRECOMPUTED))
        return set_error(MSM377_EINVAL,
                         "msm_g1_set_window_table: flags 0x%x (only EDWARDS, GLV and PRECOMPUTED select a table)",
                         flags);
    for (int k = 0; k < len; ++k)
        if (c_by_log2n[k] != 0 && (c_by_log2n[k] < 2 || c_by_log2n[k] > 20))
            return set_error(MSM377_EINVAL, "msm_g1_set_window_table: c = %d at log2 n = %d", c_by_log2n[k], k);
    const int mode = table_mode(flags);
    for (int k = 0; k < 32; ++k)
        g_ctable[mode][k].store(k < len ? c_by_log2n[k] : 0, std::memory_order_relaxed);
    return MSM377_OK;
}

extern "C" int msm_g1_set_schedule(uint32_t flags, int log2n, int c, int chunk, int sort, int reduce_log2,
                                   int groups) {
    if (flags & ~(MSM377_EDWARDS | MSM377_GLV | MSM377_PRECOMPUTED))
        return set_error(MSM377_EINVAL, "msm_g1_set_schedule: flags 0x%x (only EDWARDS, GLV and PRECOMPUTED)",
                         flags);
    if (log2n < 0 || log2n >= 32 || (c && (c < 2 || c > 20)) || (chunk && (chunk < 2 || chunk > 256)) ||
        sort < 0 || sort > 2 || (reduce_log2 && (reduce_log2 < 8 || reduce_log2 > 20)) || groups < 0 ||
        groups > kMaxGroups)
        return set_error(MSM377_EINVAL, "msm_g1_set_schedule: log2n %d c %d chunk %d sort %d reduce_log2 %d groups %d",
                         log2n, c, chunk, sort, reduce_log2, groups);
    const int mode = table_mode(flags);
    g_ctable[mode][log2n].store(c, std::memory_order_relaxed);
    g_ktable[mode][log2n].store(chunk, std::memory_order_relaxed);
    g_sorttable[mode][log2n].store(sort, std::memory_order_relaxed);
    g_rtable[mode][log2n].store(reduce_log2, std::memory_order_relaxed);
    g_gtable[mode][log2n].store(groups, std::memory_order_relaxed);
    return MSM377_OK;
}

extern "C" int msm_g1_schedule(size_t n, const msm_opts* opts, int32_t* out5) {
    if (!opts || !out5) return set_error(MSM377_EINVAL, "msm_g1_schedule: NULL argument");
    Plan p;
    if (!make_plan(n, opts, &p)) return set_error(MSM377_EINVAL, "msm_g1_schedule: bad options");
    out5[0] = p.c;
    out5[1] = p.K;
    out5[2] = p.counting ? 1 : 2;
    out5[3] = ilog2((uint64_t)p.W * p.G);
    out5[4] = p.ngroups;
    return MSM377_OK;
}

size_t msm377::msm_g1_layout_bytes(size_t n, const msm_opts* opts) {
    Plan p;
    return make_plan(n, opts, &p) ? p.total : 0;
}

// The call's own layout, or that of a smaller size whose default width is wider: the widths
// do not rise throughout (XYZZ takes 11 from 2^11 and 8 from 2^12 points, where the layout falls
// from 19.1 to 8.3 MB), and a workspace sized for the largest of a program's calls is to hold
// the smaller ones too. Within one power of two the layout still falls, by up to a sixth,
// where the pieces become longer.
extern "C" size_t msm_g1_workspace_bytes(size_t n, const msm_opts* opts) {
    Plan p, q;
    if (!make_plan(n, opts, &p)) return 0;
    size_t need = p.total;
    if (opts->c == 0 && n > 1)
        for (int k = ilog2(n); k > 0; --k) {
            const size_t below = ((size_t)1 << k) - 1;   // the largest size of the power of two below
            if (default_c(below, p.sgn, opts->flags) > p.c && make_plan(below, opts, &q) && q.total > need)
                need = q.total;
        }
    return need;
}

extern "C" size_t msm_points_prepared_bytes(size_t n, uint32_t flags) {
    if (flags & ~(MSM377_EDWARDS | MSM377_GLV)) return 0;
    if (n >= (1ull << 30)) return 0;
    return stored_count(n, flags) * 16 * (size_t)stored_vec(flags);
}

extern "C" int msm_points_prepare_ex(const uint32_t* points_std, size_t n, uint32_t* out, uint32_t flags,
                                     void* stream) {
    if (flags & ~(MSM377_EDWARDS | MSM377_GLV))
        return set_error(MSM377_EINVAL, "msm_points_prepare_ex: flags 0x%x (only EDWARDS and GLV)", flags);
    if (n >= (1ull << 30)) return set_error(MSM377_EINVAL, "msm_points_prepare_ex: n = %zu too large", n);
    if (n == 0) return MSM377_OK;
    if (!points_std || !out || !aligned(points_std, 16) || !aligned(out, 16))
        return set_error(MSM377_EINVAL, "msm_points_prepare_ex: null or non-16-byte-aligned pointer");
    launch_prepare(reinterpret_cast<const uint4*>(points_std), reinterpret_cast<uint4*>(out), n, flags,
                   as_stream(stream));
    return check_launch("msm_points_prepare_ex");
}

extern "C" int msm_points_prepare(const uint32_t* points_std, size_t n, uint32_t* out, void* stream) {
    return msm_points_prepare_ex(points_std, n, out, 0, stream);
}

extern "C" size_t msm_points_precomputed_bytes(size_t n, const msm_opts* opts) {
    if (!opts || !(opts->flags & MSM377_PRECOMPUTED)) return 0;
    msm_opts o = *opts;
    o.flags |= MSM377_POINTS_PREPARED;
    Plan p;
    if (!make_plan(n, &o, &p)) return 0;
    return p.items * 16 * (size_t)ModelEdwards::kStored;
}

extern "C" int msm_points_precompute(const uint32_t* points_std, size_t n, uint32_t* out, const msm_opts* opts) {
    if (!opts) return set_error(MSM377_EINVAL, "msm_points_precompute: opts is NULL");
    if (msm_points_precomputed_bytes(n > 0 ? n : 1, opts) == 0)  // options valid (n = 0 needs 0 bytes)
        return set_error(MSM377_EINVAL,
                         "msm_points_precompute: needs MSM377_EDWARDS | MSM377_PRECOMPUTED, an explicit c and "
                         "valid options (c=%d scalar_bits=%d)", opts->c, opts->scalar_bits);
    if (n == 0) return MSM377_OK;
    if (!points_std || !out || !aligned(points_std, 16) || !aligned(out, 16))
        return set_error(MSM377_EINVAL, "msm_points_precompute: null or non-16-byte-aligned pointer");
    msm_opts o = *opts;
    o.flags |= MSM377_POINTS_PREPARED;
    Plan p;
    make_plan(n, &o, &p);
    cudaStream_t s = as_stream(opts->stream);
    const size_t threads = (p.np + kEdChunk - 1) / kEdChunk;  // whole warps: grid_for rounds up to 128
    k_precompute_ed<<<grid_for(threads, 128), 128, 0, s>>>(reinterpret_cast<const uint4*>(points_std),
                                                           reinterpret_cast<uint4*>(out), n, p.np, p.c, p.Wd);
    note_launches(1);
    return check_launch("msm_points_precompute");
}

namespace {

// Phase 1-3 of one MSM on stream s: counters reset, preparation, digits, sort, and the
// pieces of every window group. Fills `job` with what the accumulations and tails need.
// reset_status = false: the caller has cleared the status word and the counters
// already (msm_g1_host validates point chunks on a helper stream first).
struct Job {
    const uint4* pts;
    const uint32_t* items;
};

PieceArgs piece_args(const Plan& p, void* workspace, int g) {
    PieceArgs a;
    a.start = at<uint32_t>(workspace, p.off_bins);
    a.nb = p.Bp + 1;
    a.Bp = p.Bp;
    a.w0 = g * p.gw;
    a.nwin = p.W - a.w0 < p.gw ? p.W - a.w0 : p.gw;
    a.total = (uint32_t)((size_t)(a.w0 + a.nwin) * p.items);
    a.cap = (uint32_t)p.K;
    a.cap_few = (uint32_t)p.K_few;
    a.nonzero = p.K_few < p.K ? at<uint32_t>(workspace, p.off_ctrl) + kNonzero : nullptr;
    a.all = (uint32_t)((size_t)p.W * p.items);
    a.group_items = (uint32_t)((size_t)p.gw * p.items);
    a.wave = (uint32_t)p.wave;
    a.shared = (uint32_t)p.shared;
    a.levels = p.levels;
    a.small_parts = p.small_parts;
    a.ctrl = at<uint32_t>(workspace, p.off_ctrl) + (size_t)g * kCtrlWords;
    a.pieces = at<uint4>(workspace, p.off_pieces) + (size_t)g * p.max_pieces;
    a.small = at<uint4>(workspace, p.off_small) + (size_t)g * p.max_small;
    for (int k = 0; k < 3; ++k) a.tree[k] = at<uint4>(workspace, p.off_tree[k]) + (size_t)g * p.max_tree[k];
    a.buckets = at<uint4>(workspace, p.off_buckets);
    return a;
}

AccArgs acc_args(const Plan& p, const Job& job, void* workspace, int g) {
    const PieceArgs pa = piece_args(p, workspace, g);
    AccArgs a;
    a.items = job.items;
    a.pts = job.pts;
    a.npts = (uint32_t)p.items;   // stored rows: np, or Wd np with precomputed copies
    a.buckets = pa.buckets;
    a.parts = at<uint4>(workspace, p.off_parts) + (size_t)g * p.max_parts * kXyzzVec;
    a.pieces = pa.pieces;
    a.hist = pa.ctrl + kHist;
    a.cap = pa.cap;
    return a;
}

int enqueue_head(const Plan& p, const uint32_t* points, const uint32_t* scalars, void* workspace,
                 const msm_opts* opts, cudaStream_t s, Job* job, bool reset_status = true) {
    const size_t n = p.n;
    int* status = at<int>(workspace, p.off_status);
    if (reset_status)
        MSM_CUDA_TRY(cudaMemsetAsync(status, 0, p.ctrl_bytes, s));
    const uint4* pts = reinterpret_cast<const uint4*>(points);
    if ((opts->flags & MSM377_VALIDATE) && !(opts->flags & MSM377_POINTS_PREPARED)) {
        const int r = launch_validate(points, n, (opts->flags & (MSM377_EDWARDS | MSM377_GLV)) != 0, status, s);
        if (r) return r;
    }
    if (!(opts->flags & MSM377_POINTS_PREPARED)) {
        uint4* prep = at<uint4>(workspace, p.off_points);
        launch_prepare(pts, prep, n, opts->flags, s);
        pts = prep;
    }
    const size_t np = p.items;  // items per pipeline window
    uint32_t* keys[2] = {at<uint32_t>(workspace, p.off_keys0), at<uint32_t>(workspace, p.off_keys1)};
    uint32_t* vals[2] = {at<uint32_t>(workspace, p.off_vals0), at<uint32_t>(workspace, p.off_vals1)};
    const PieceArgs pieces = piece_args(p, workspace, 0);
    const auto digits = pieces.nonzero ? k_digits<true> : k_digits<false>;
    digits<<<grid_for(n, kDigitThreads), kDigitThreads, 0, s>>>(reinterpret_cast<const uint4*>(scalars), n, p.c, p.Wd,
                                                                p.sgn, p.user_bits, p.glv, keys[0], status,
                                                                pieces.ctrl + kNonzero);
    note_launches(1);
    int cur = 0;
    bool pieces_counted = false;
    const int pre_w = p.pre ? p.Wd : 0;
    const uint32_t nb = p.Bp + 1;
    uint32_t* bins = at<uint32_t>(workspace, p.off_bins);
    if (p.counting) {
        // counting sort: count, scan, scatter (window-major bins, window w at w np)
        const size_t total = (size_t)p.W * np;
        uint32_t* bsum = at<uint32_t>(workspace, p.off_bsum);
        uint32_t* rank = at<uint32_t>(workspace, p.off_rank);
        const dim3 gw(grid_for(np, 256), (unsigned)p.W);
        uint32_t* tcnt = at<uint32_t>(workspace, p.off_tcnt);
        if (p.ttiles) {
            // the counters of one block exceed the default 48 KB of dynamic shared memory
            const size_t smem = (size_t)((nb + 1) / 2) * 4;
            MSM_CUDA_TRY(cudaFuncSetAttribute(k_tile_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kTileSmemMax));
            k_tile_count<<<dim3(p.ttiles, (unsigned)p.W), kTileThreads, smem, s>>>(keys[0], np, nb, p.tT, p.ttiles,
                                                                                  tcnt, rank);
            pieces_counted = p.ngroups == 1;
            k_tile_totals<<<grid_for(p.nbins, kBinBlock), kBinBlock, 0, s>>>(
                tcnt, nb, p.ttiles, (uint32_t)p.W, bins, bsum, pieces, pieces_counted ? 1 : 0);
            k_tile_offsets<<<grid_for(p.nbins, 256), 256, 0, s>>>(tcnt, nb, p.ttiles, (uint32_t)p.W, bins, bsum);
            k_tile_scatter<<<gw, 256, 0, s>>>(keys[0], rank, vals[0], total, np, nb, p.tT, p.ttiles, tcnt, p.np, pre_w);
            note_launches(4);
        } else {
            const size_t ntiles = (p.nbins + kScanTile - 1) / kScanTile;
            MSM_CUDA_TRY(cudaMemsetAsync(bins, 0, p.nbins * 4, s));
            k_bin_count<<<gw, 256, 0, s>>>(keys[0], np, nb, bins, rank);
            k_scan_tiles<<<(unsigned)ntiles, kScanBlock, 0, s>>>(bins, p.nbins, bsum);
            k_scan_totals<<<1, kScanBlock, 0, s>>>(bsum, ntiles);
            k_scan_add<<<grid_for(p.nbins, 256), 256, 0, s>>>(bins, p.nbins, bsum);
            k_bin_scatter<<<gw, 256, 0, s>>>(keys[0], rank, vals[0], total, np, nb, bins, p.np, pre_w);
            note_launches(5);
        }
    } else {
        uint32_t* hist = at<uint32_t>(workspace, p.off_hist);
        uint32_t* dtot = at<uint32_t>(workspace, p.off_dtot);
        for (int pass = 0; pass < p.passes; ++pass) {
            const int shift = p.rb * pass;
            const dim3 g((unsigned)p.tiles, (unsigned)p.W);
            k_sort_hist<8><<<g, kSortThreads, 0, s>>>(keys[cur], np, shift, p.tiles, hist);
            k_sort_scan_tiles<8><<<dim3(1u << 8, p.W), kSortThreads, 0, s>>>(hist, p.tiles, dtot);
            k_sort_scan_digits<8><<<p.W, kSortThreads, 0, s>>>(dtot);
            k_sort_scatter<8><<<g, kSortThreads, 0, s>>>(keys[cur], pass ? vals[cur] : nullptr, keys[cur ^ 1],
                                                         vals[cur ^ 1], np, shift, p.tiles, hist, dtot, p.np, pre_w);
            note_launches(4);
            cur ^= 1;
        }
        k_run_starts<<<dim3(grid_for(np, kStartThreads), (unsigned)p.W), kStartThreads, 0, s>>>(keys[cur], np, nb, bins);
        note_launches(1);
    }
    job->pts = pts;
    job->items = vals[cur];
    for (int g = 0; g < p.ngroups; ++g) {
        const PieceArgs a = piece_args(p, workspace, g);
        const unsigned grid = grid_for((size_t)a.nwin * nb, kPieceThreads);
        if (!pieces_counted) {
            k_piece_count<<<grid, kPieceThreads, 0, s>>>(a);
            note_launches(1);
        }
        k_piece_emit<<<grid, kPieceThreads, 0, s>>>(a);
        note_launches(1);
    }
    return check_launch("msm head");
}

// Phase 5-6 and the per-window sums of stage 7 for the windows of group g on stream s:
// partial merges, bucket reduction, and S_w for each window, in the group's buffers.
template <class M>
int enqueue_group_tail_m(const Plan& p, const AccArgs& acc, int g, void* workspace, cudaStream_t s) {
    int* S = at<int>(workspace, p.off_S);
    const PieceArgs a = piece_args(p, workspace, g);
    // 5. the parts of buckets cut into pieces
    for (int lv = 0; lv < p.levels; ++lv) {
        const size_t want = p.max_tree[lv] + (lv == 0 ? (p.max_small + kTreeThreads - 1) / kTreeThreads : 0);
        k_merge_parts<M><<<(unsigned)(want < kTreeWave ? want : kTreeWave), kTreeThreads, 0, s>>>(
            acc.parts, acc.buckets, a.tree[lv], a.ctrl + kNTree + lv, lv == 0 ? a.small : nullptr,
            lv == 0 ? a.ctrl + kNSmall : nullptr);
        note_launches(1);
    }
    // 6. bucket reduction of the group's windows
    const size_t nseg = (size_t)a.nwin * (p.logG + 2);
    uint4* P0 = at<uint4>(workspace, p.off_P0) + (size_t)g * p.gw * (p.logG + 2) * p.nb * kXyzzVec;
    uint4* Z = P0;
    if (p.L > 1) {
        const size_t yv = (size_t)p.gw * p.G * kXyzzVec;
        uint4* Y = at<uint4>(workspace, p.off_Y) + (size_t)g * yv;
        uint4* V = at<uint4>(workspace, p.off_V) + (size_t)g * yv;
        const size_t nt = (size_t)a.nwin * p.G;
        if (p.pairs)
            k_reduce_pairs<M><<<grid_for(2 * nt, 128), 128, 0, s>>>(a.buckets, p.Bp, p.L, a.w0, a.nwin, p.G, Y, V);
        else
            k_reduce_segments<M><<<grid_for(nt, 128), 128, 0, s>>>(a.buckets, p.Bp, p.L, a.w0, a.nwin, p.G, Y, V);
        k_bit_sums<M, false><<<(unsigned)(nseg * p.nb), kTreeThreads, 0, s>>>(Y, V, a.nwin, p.G, p.logG, p.nb, P0);
        note_launches(2);
    } else {
        const uint4* B = a.buckets + (size_t)a.w0 * p.Bp * kXyzzVec;
        k_bit_sums<M, true><<<(unsigned)(nseg * p.nb), kTreeThreads, 0, s>>>(B, B, a.nwin, p.G, p.logG, p.nb, P0);
        note_launches(1);
    }
    if (p.nb > 1) {
        Z = at<uint4>(workspace, p.off_P1) + (size_t)g * p.gw * (p.logG + 2) * kXyzzVec;
        k_sum_rows<M><<<(unsigned)nseg, kTreeThreads, 0, s>>>(P0, p.nb, Z);
        note_launches(1);
    }
    // 7a. the per-window sums S_w
    k_window_horner_w<M><<<(unsigned)a.nwin, 128, 0, s>>>(Z, a.nwin, p.logG, p.log2L, S + (size_t)a.w0 * wred::kLimbPointWords);
    note_launches(1);
    return check_launch("msm tail");
}

int enqueue_group_tail(const Plan& p, const AccArgs& a, int g, void* workspace, cudaStream_t s) {
    return p.edw ? enqueue_group_tail_m<ModelEdwards>(p, a, g, workspace, s)
                 : enqueue_group_tail_m<ModelXyzz>(p, a, g, workspace, s);
}

// 7b. the window combination and normalisation into out.
int enqueue_chain(const Plan& p, void* workspace, uint32_t* out, cudaStream_t s) {
    const int* S = at<int>(workspace, p.off_S);
    if (p.edw)
        k_chain_w<ModelEdwards><<<1, 128, 0, s>>>(S, p.W, p.c, out);
    else
        k_chain_w<ModelXyzz><<<1, 128, 0, s>>>(S, p.W, p.c, out);
    note_launches(1);
    return check_launch("msm chain");
}

// Phase 5-7 of one MSM as a single window group on stream s (batched calls).
int enqueue_tail(const Plan& p, const AccArgs& a, void* workspace, uint32_t* out, cudaStream_t s) {
    int r = enqueue_group_tail(p, a, 0, workspace, s);
    if (r) return r;
    return enqueue_chain(p, workspace, out, s);
}

// Accumulation of one window group.
int enqueue_accumulate(const Plan& p, const AccArgs& a, cudaStream_t s) {
    const unsigned grid = grid_for(p.max_pieces, 128);
    if (p.edw)
        k_accumulate<ModelEdwards><<<grid, 128, 0, s>>>(a);
    else
        k_accumulate<ModelXyzz><<<grid, 128, 0, s>>>(a);
    note_launches(1);
    return check_launch("msm accumulate");
}

// A helper stream of the highest priority and events, one set per caller stream
// (so calls on different streams never share them), created on first use.
struct Overlap {
    cudaStream_t hi;
    cudaEvent_t ev[kMaxGroups + 1];
};
constexpr int kOverlapSlots = 32;
struct OverlapSlot {
    bool used = false;
    int dev = -1;
    cudaStream_t caller = nullptr;
    Overlap ov;
};
OverlapSlot g_overlap[kOverlapSlots];
std::mutex g_overlap_mu;

// nullptr when every slot is taken: the groups then run in sequence on s.
const Overlap* overlap_for(cudaStream_t s) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(g_overlap_mu);
    for (auto& sl : g_overlap)
        if (sl.used && sl.dev == dev && sl.caller == s) return &sl.ov;
    for (auto& sl : g_overlap) {
        if (sl.used) continue;
        int least = 0, greatest = 0;
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) return nullptr;
        if (cudaStreamCreateWithPriority(&sl.ov.hi, cudaStreamNonBlocking, greatest) != cudaSuccess) return nullptr;
        for (int i = 0; i <= kMaxGroups; ++i)
            if (cudaEventCreateWithFlags(&sl.ov.ev[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
        sl.used = true;
        sl.dev = dev;
        sl.caller = s;
        return &sl.ov;
    }
    return nullptr;
}

// Phase 4-7 on stream s: the accumulation group by group, each group's tail on the
// high-priority helper as soon as its accumulation is done (overlapping the next
// group's accumulation), then the window chain on s. Without a helper (ov null, or
// one group) everything runs in order on s. prof: stage marks after the last
// accumulation and after the chain.
int enqueue_body(const Plan& p, const Job& job, void* workspace, uint32_t* out, cudaStream_t s, const Overlap* ov,
                 bool prof) {
    int r;
    if (p.ngroups <= 1 || !ov) {
        for (int g = 0; g < p.ngroups; ++g)
            if ((r = enqueue_accumulate(p, acc_args(p, job, workspace, g), s))) return r;
        if (prof) profile_mark(s);
        for (int g = 0; g < p.ngroups; ++g)
            if ((r = enqueue_group_tail(p, acc_args(p, job, workspace, g), g, workspace, s))) return r;
    } else {
        for (int g = 0; g < p.ngroups; ++g) {
            const AccArgs a = acc_args(p, job, workspace, g);
            if ((r = enqueue_accumulate(p, a, s))) return r;
            MSM_CUDA_TRY(cudaEventRecord(ov->ev[g], s));
            MSM_CUDA_TRY(cudaStreamWaitEvent(ov->hi, ov->ev[g], 0));
            if ((r = enqueue_group_tail(p, a, g, workspace, ov->hi))) return r;
        }
        if (prof) profile_mark(s);
        MSM_CUDA_TRY(cudaEventRecord(ov->ev[kMaxGroups], ov->hi));
        MSM_CUDA_TRY(cudaStreamWaitEvent(s, ov->ev[kMaxGroups], 0));
    }
    if ((r = enqueue_chain(p, workspace, out, s))) return r;
    if (prof) profile_mark(s);
    return MSM377_OK;
}

// Library-owned helper streams for batched calls, per device, created once.
constexpr int kMaxDevices = 64;
constexpr int kAuxStreams = 16;
constexpr int kHostChunks = 4;  // the copy (about 200 GB/s) is shorter than the preparation; small first chunk
constexpr size_t kSplitPrepMin = size_t(1) << 15;  // msm_g1: prepare beside the head from this size on
static_assert(1 + kHostChunks <= kAuxStreams, "msm_g1_host needs a copy stream and one stream per chunk");
struct DeviceAux {
    bool ready = false;
    int sms = 0, acc_blocks_per_sm[2] = {0, 0};  // k_accumulate_batched per model
    cudaStream_t st[kAuxStreams];
    cudaEvent_t fork, done[kAuxStreams];
    cudaEvent_t chunk[kHostChunks];  // msm_g1_host: point chunk k has arrived
};
DeviceAux g_aux[kMaxDevices];
std::mutex g_aux_mu;

int device_aux(DeviceAux** out) {
    int dev = 0;
    MSM_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return set_error(MSM377_EINVAL, "device ordinal %d out of range", dev);
    std::lock_guard<std::mutex> lock(g_aux_mu);
    DeviceAux& a = g_aux[dev];
    if (!a.ready) {
        MSM_CUDA_TRY(cudaDeviceGetAttribute(&a.sms, cudaDevAttrMultiProcessorCount, dev));
        MSM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a.acc_blocks_per_sm[0],
                                                                   k_accumulate_batched<ModelXyzz>, 128, 0));
        MSM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a.acc_blocks_per_sm[1],
                                                                   k_accumulate_batched<ModelEdwards>, 128, 0));
        for (int m = 0; m < 2; ++m)
            if (a.acc_blocks_per_sm[m] < 1) a.acc_blocks_per_sm[m] = 1;
        for (int i = 0; i < kAuxStreams; ++i) {
            MSM_CUDA_TRY(cudaStreamCreateWithFlags(&a.st[i], cudaStreamNonBlocking));
            MSM_CUDA_TRY(cudaEventCreateWithFlags(&a.done[i], cudaEventDisableTiming));
        }
        MSM_CUDA_TRY(cudaEventCreateWithFlags(&a.fork, cudaEventDisableTiming));
        for (int k = 0; k < kHostChunks; ++k) MSM_CUDA_TRY(cudaEventCreateWithFlags(&a.chunk[k], cudaEventDisableTiming));
        a.ready = true;
    }
    *out = &a;
    return MSM377_OK;
}

// Helper streams wait for work already on s; then s waits for the helpers.
int fork_from(DeviceAux* aux, cudaStream_t s, int k) {
    MSM_CUDA_TRY(cudaEventRecord(aux->fork, s));
    for (int i = 0; i < k; ++i) MSM_CUDA_TRY(cudaStreamWaitEvent(aux->st[i], aux->fork, 0));
    return MSM377_OK;
}
int join_into(DeviceAux* aux, cudaStream_t s, int k) {
    for (int i = 0; i < k; ++i) {
        MSM_CUDA_TRY(cudaEventRecord(aux->done[i], aux->st[i]));
        MSM_CUDA_TRY(cudaStreamWaitEvent(s, aux->done[i], 0));
    }
    return MSM377_OK;
}

}  // namespace

namespace msm377 {

int msm_g1_run(const uint32_t* points, const uint32_t* scalars, size_t n, uint32_t* out, void* workspace,
               size_t workspace_bytes, const msm_opts* opts, bool overlap) {
    if (!opts) return set_error(MSM377_EINVAL, "msm_g1: opts is NULL");
    if (!out) return set_error(MSM377_EINVAL, "msm_g1: out is NULL");
    cudaStream_t s = as_stream(opts->stream);
    Plan p;
    if (!make_plan(n, opts, &p))
        return set_error(MSM377_EINVAL, "msm_g1: bad options (c=%d scalar_bits=%d) or n too large",
                         opts->c, opts->scalar_bits);
    if (!workspace || !aligned(workspace, 256))
        return set_error(MSM377_EINVAL, "msm_g1: workspace NULL or not 256-byte aligned");
    if (workspace_bytes < p.total)
        return set_error(MSM377_ENOMEM, "msm_g1: workspace %zu bytes, need %zu", workspace_bytes, p.total);
    if ((opts->flags & MSM377_VALIDATE) && (opts->flags & MSM377_POINTS_PREPARED))
        return set_error(MSM377_EINVAL, "msm_g1: MSM377_VALIDATE checks standard-form input points; stored "
                         "(prepared) points are validated when the set is made (msm_points_create)");
    const bool prof = (opts->flags & MSM377_PROFILE) != 0;
    if (prof) {
        int pr = profile_begin(s);
        if (pr) return pr;
    }
    if (n == 0) {
        MSM_CUDA_TRY(cudaMemsetAsync(at<int>(workspace, p.off_status), 0, sizeof(int), s));
        MSM_CUDA_TRY(cudaMemsetAsync(out, 0, 24 * sizeof(uint32_t), s));
        return MSM377_OK;
    }
    if (!points || !scalars || !aligned(points, 16) || !aligned(scalars, 16))
        return set_error(MSM377_EINVAL, "msm_g1: points/scalars NULL or not 16-byte aligned");
    Job job;
    // Standard-form points: their preparation (and validation) runs on the caller
    // stream's high-priority helper while the digits and the sort, which need only
    // the scalars, run on s; the accumulation waits for both.
    const bool split = overlap && !prof && !(opts->flags & MSM377_POINTS_PREPARED) && n >= kSplitPrepMin;
    const Overlap* ov = (overlap && (p.ngroups > 1 || split)) ? overlap_for(s) : nullptr;
    int r;
    if (split && ov) {
        int* status = at<int>(workspace, p.off_status);
        MSM_CUDA_TRY(cudaMemsetAsync(status, 0, p.ctrl_bytes, s));
        MSM_CUDA_TRY(cudaEventRecord(ov->ev[0], s));
        MSM_CUDA_TRY(cudaStreamWaitEvent(ov->hi, ov->ev[0], 0));
        if (opts->flags & MSM377_VALIDATE) {
            r = launch_validate(points, n, (opts->flags & (MSM377_EDWARDS | MSM377_GLV)) != 0, status, ov->hi);
            if (r) return r;
        }
        uint4* prep = at<uint4>(workspace, p.off_points);
        launch_prepare(reinterpret_cast<const uint4*>(points), prep, n, opts->flags, ov->hi);
        MSM_CUDA_TRY(cudaEventRecord(ov->ev[1], ov->hi));
        msm_opts op = *opts;
        op.flags |= MSM377_POINTS_PREPARED;  // the plan keeps the prepared region in the workspace
        r = enqueue_head(p, reinterpret_cast<const uint32_t*>(prep), scalars, workspace, &op, s, &job, false);
        if (r) return r;
        MSM_CUDA_TRY(cudaStreamWaitEvent(s, ov->ev[1], 0));
    } else {
        r = enqueue_head(p, points, scalars, workspace, opts, s, &job);
        if (r) return r;
    }
    if (prof) profile_mark(s);
    return enqueue_body(p, job, workspace, out, s, p.ngroups > 1 ? ov : nullptr, prof);
}

}  // namespace msm377

extern "C" int msm_g1(const uint32_t* points, const uint32_t* scalars, size_t n, uint32_t* out,
                      void* workspace, size_t workspace_bytes, const msm_opts* opts) {
    return msm_g1_run(points, scalars, n, out, workspace, workspace_bytes, opts, true);
}

namespace {
constexpr size_t kBatchHeader = 256;

// c for job i of a batch: the job's own, else the options', else the size default.
bool batch_plans(const msm_job* jobs, size_t njobs, const msm_opts* opts, Plan* plans, size_t* total) {
    size_t off = kBatchHeader, items = 0;
    const bool glv = (opts->flags & MSM377_GLV) != 0;
    const int sgn = opts->signed_digits ? 1 : 0, bits = glv ? 127 : (opts->scalar_bits > 0 ? opts->scalar_bits : 256);
    for (size_t i = 0; i < njobs; ++i) {   // about; the plans check their options
        const int own = jobs[i].c ? jobs[i].c : opts->c;
        const int c = own > 0 ? own : default_c(jobs[i].n, sgn, opts->flags, false);
        items += (size_t)((bits + sgn + c - 1) / c) * (glv ? 2 : 1) * jobs[i].n;
    }
    for (size_t i = 0; i < njobs; ++i) {
        msm_opts o = *opts;
        if (jobs[i].c) o.c = jobs[i].c;
        if (!make_plan(jobs[i].n, &o, &plans[i], false, items)) return false;
        off += align_up(plans[i].total, 256);
    }
    *total = off;
    return true;
}
}  // namespace

extern "C" size_t msm_g1_batched_workspace_bytes(const msm_job* jobs, size_t njobs, const msm_opts* opts) {
    if (!jobs || !opts || njobs == 0 || njobs > (size_t)kMaxBatch) return 0;
    Plan plans[kMaxBatch];
    size_t total = 0;
    if (!batch_plans(jobs, njobs, opts, plans, &total)) return 0;
    return total;
}

extern "C" int msm_g1_batched(const msm_job* jobs, size_t njobs, void* workspace, size_t workspace_bytes,
                              const msm_opts* opts) {
    if (!jobs || !opts) return set_error(MSM377_EINVAL, "msm_g1_batched: NULL argument");
    if (njobs == 0) return MSM377_OK;
    if (njobs > (size_t)kMaxBatch)
        return set_error(MSM377_EINVAL, "msm_g1_batched: %zu jobs, at most %d per call", njobs, kMaxBatch);
    if (opts->flags & (MSM377_PROFILE | MSM377_VALIDATE))
        return set_error(MSM377_EINVAL, "msm_g1_batched: MSM377_PROFILE and MSM377_VALIDATE are not supported "
                         "(validate point sets once with msm_points_validate or msm_points_create)");
    Plan plans[kMaxBatch];
    size_t total = 0;
    if (!batch_plans(jobs, njobs, opts, plans, &total))
        return set_error(MSM377_EINVAL, "msm_g1_batched: bad options or n too large in some job");
    if (!workspace || !aligned(workspace, 256))
        return set_error(MSM377_EINVAL, "msm_g1_batched: workspace NULL or not 256-byte aligned");
    if (workspace_bytes < total)
        return set_error(MSM377_ENOMEM, "msm_g1_batched: workspace %zu bytes, need %zu", workspace_bytes, total);
    for (size_t i = 0; i < njobs; ++i) {
        if (!jobs[i].out) return set_error(MSM377_EINVAL, "msm_g1_batched: job %zu has no output", i);
        if (jobs[i].n && (!jobs[i].points || !jobs[i].scalars || !aligned(jobs[i].points, 16) ||
                          !aligned(jobs[i].scalars, 16)))
            return set_error(MSM377_EINVAL, "msm_g1_batched: job %zu points/scalars NULL or misaligned", i);
    }
    DeviceAux* aux = nullptr;
    int r = device_aux(&aux);
    if (r) return r;
    cudaStream_t s = as_stream(opts->stream);
    const int nst = njobs < (size_t)kAuxStreams ? (int)njobs : kAuxStreams;

    // heads of all jobs on the helper streams
    BatchAcc b;
    b.njobs = 0;
    b.prefix[0] = 0;
    uint32_t* counter = static_cast<uint32_t*>(workspace);
    MSM_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(uint32_t), s));
    r = fork_from(aux, s, nst);
    if (r) return r;
    char* base = static_cast<char*>(workspace) + kBatchHeader;
    void* ws[kMaxBatch];
    for (size_t i = 0; i < njobs; ++i) {
        ws[i] = base;
        base += align_up(plans[i].total, 256);
        cudaStream_t si = aux->st[i % nst];
        if (jobs[i].n == 0) {
            MSM_CUDA_TRY(cudaMemsetAsync(jobs[i].out, 0, 24 * sizeof(uint32_t), si));
            continue;
        }
        Job job;
        r = enqueue_head(plans[i], jobs[i].points, jobs[i].scalars, ws[i], opts, si, &job);
        if (r) return r;
        b.job[b.njobs] = acc_args(plans[i], job, ws[i], 0);
        b.prefix[b.njobs + 1] = b.prefix[b.njobs] + (uint32_t)((plans[i].max_pieces + 31) / 32 * 32);
        ++b.njobs;
    }
    r = join_into(aux, s, nst);
    if (r) return r;

    // every job's bucket accumulation in one persistent launch
    if (b.njobs > 0) {
        b.counter = counter;
        const int edw = (opts->flags & MSM377_EDWARDS) ? 1 : 0;
        const unsigned grid = (unsigned)(aux->sms * aux->acc_blocks_per_sm[edw]);
        if (edw)
            k_accumulate_batched<ModelEdwards><<<grid, 128, 0, s>>>(b);
        else
            k_accumulate_batched<ModelXyzz><<<grid, 128, 0, s>>>(b);
        note_launches(1);
        r = check_launch("msm_g1_batched accumulate");
        if (r) return r;
    }

    // tails of all jobs on the helper streams
    r = fork_from(aux, s, nst);
    if (r) return r;
    for (size_t i = 0, k = 0; i < njobs; ++i) {
        if (jobs[i].n == 0) continue;
        r = enqueue_tail(plans[i], b.job[k], ws[i], jobs[i].out, aux->st[i % nst]);
        if (r) return r;
        ++k;
    }
    return join_into(aux, s, nst);
}

extern "C" int msm_g1_status(const void* workspace, const msm_opts* opts) {
    if (!workspace || !opts) return set_error(MSM377_EINVAL, "msm_g1_status: NULL argument");
    int st = 0;
    cudaStream_t s = as_stream(opts->stream);
    MSM_CUDA_TRY(cudaMemcpyAsync(&st, workspace, sizeof(int), cudaMemcpyDeviceToHost, s));
    MSM_CUDA_TRY(cudaStreamSynchronize(s));
    if (st == MSM377_ERANGE) return set_error(MSM377_ERANGE, "msm_g1: a scalar exceeds scalar_bits");
    if (st == MSM377_ENOTONCURVE)
        return set_error(MSM377_ENOTONCURVE, "msm_g1: an input point is not on the curve (or, with "
                         "MSM377_EDWARDS / MSM377_GLV, not in the order-r subgroup)");
    return st;
}

namespace {
// A layout of `core` bytes with the copied points, scalars and the result behind it.
size_t host_bytes(size_t core, size_t n) { return core + align_up(n * 96, 256) + align_up(n * 32, 256) + 256; }
}  // namespace

extern "C" size_t msm_g1_host_workspace_bytes(size_t n, const msm_opts* opts) {
    if (!opts) return 0;
    msm_opts o = *opts;
    o.flags &= ~MSM377_POINTS_PREPARED;
    size_t core = msm_g1_workspace_bytes(n, &o);
    if (!core) return 0;
    return host_bytes(core, n);
}

extern "C" int msm_g1_host(const uint32_t* points_host, const uint32_t* scalars_host, size_t n,
                           uint32_t* out_host, void* workspace, size_t workspace_bytes,
                           const msm_opts* opts) {
    if (!opts || !out_host || !workspace) return set_error(MSM377_EINVAL, "msm_g1_host: NULL argument");
    if (n && (!points_host || !scalars_host)) return set_error(MSM377_EINVAL, "msm_g1_host: NULL inputs");
    msm_opts o = *opts;
    o.flags &= ~(MSM377_POINTS_PREPARED | MSM377_PROFILE);
    Plan p;
    if (!make_plan(n, &o, &p)) return set_error(MSM377_EINVAL, "msm_g1_host: bad options");
    const size_t core = p.total, need = host_bytes(core, n);
    if (workspace_bytes < need)
        return set_error(MSM377_ENOMEM, "msm_g1_host: workspace %zu bytes, need %zu", workspace_bytes, need);
    if (!aligned(workspace, 256)) return set_error(MSM377_EINVAL, "msm_g1_host: workspace not 256-byte aligned");
    char* base = static_cast<char*>(workspace);
    uint32_t* d_pts = reinterpret_cast<uint32_t*>(base + core);
    uint32_t* d_sc = reinterpret_cast<uint32_t*>(base + core + align_up(n * 96, 256));
    uint32_t* d_out = reinterpret_cast<uint32_t*>(base + core + align_up(n * 96, 256) + align_up(n * 32, 256));
    cudaStream_t s = as_stream(o.stream);
    if (n == 0) {
        int r = msm_g1(d_pts, d_sc, 0, d_out, workspace, core, &o);
        if (r) return r;
        MSM_CUDA_TRY(cudaMemcpyAsync(out_host, d_out, 24 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
        return msm_g1_status(workspace, &o);
    }
    // The points travel in chunks on one helper stream and each chunk is prepared
    // on a helper stream of its own as soon as it has arrived (the chunks' launches
    // are sized to fill the GPU together), while the scalars' copy, digits and
    // bucket sort run on the caller's stream; the accumulation waits for them all.
    DeviceAux* aux = nullptr;
    int r = device_aux(&aux);
    if (r) return r;
    cudaStream_t sc = aux->st[0];
    MSM_CUDA_TRY(cudaMemsetAsync(at<int>(workspace, p.off_status), 0, p.ctrl_bytes, s));  // before the fork
    r = fork_from(aux, s, 1 + kHostChunks);
    if (r) return r;
    uint4* prep = at<uint4>(workspace, p.off_points);
    const size_t per = (n + kHostChunks - 1) / kHostChunks;
    for (int k = 0; k < kHostChunks; ++k) {
        const size_t a = (size_t)k * per, b = a + per < n ? a + per : n;
        if (a >= b) break;
        cudaStream_t sp = aux->st[1 + k];
        MSM_CUDA_TRY(cudaMemcpyAsync(d_pts + 24 * a, points_host + 24 * a, (b - a) * 96, cudaMemcpyHostToDevice, sc));
        MSM_CUDA_TRY(cudaEventRecord(aux->chunk[k], sc));
        MSM_CUDA_TRY(cudaStreamWaitEvent(sp, aux->chunk[k], 0));
        if (o.flags & MSM377_VALIDATE) {
            r = launch_validate(d_pts + 24 * a, b - a, (o.flags & (MSM377_EDWARDS | MSM377_GLV)) != 0,
                                at<int>(workspace, p.off_status), sp);
            if (r) return r;
        }
        launch_prepare_range(reinterpret_cast<const uint4*>(d_pts), prep, n, a, b, o.flags, sp, n);
    }
    MSM_CUDA_TRY(cudaMemcpyAsync(d_sc, scalars_host, n * 32, cudaMemcpyHostToDevice, s));
    msm_opts op = o;
    op.flags |= MSM377_POINTS_PREPARED;  // the plan above keeps the prepared region in the workspace
    Job job;
    r = enqueue_head(p, reinterpret_cast<const uint32_t*>(prep), d_sc, workspace, &op, s, &job, false);
    if (r) return r;
    r = join_into(aux, s, 1 + kHostChunks);
    if (r) return r;
    r = enqueue_body(p, job, workspace, d_out, s, p.ngroups > 1 ? overlap_for(s) : nullptr, false);
    if (r) return r;
    MSM_CUDA_TRY(cudaMemcpyAsync(out_host, d_out, 24 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    return msm_g1_status(workspace, &o);
}
