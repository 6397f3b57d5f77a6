// Point arithmetic spread over a block of four warps, for latency-bound chains of
// point operations (the window combination, the per-window sums, padd_chain): one
// accumulator is updated again and again, so a chain costs the latency of its
// products, not their number.
//
// One product runs on the 32 lanes of a warp. A field element is held as 15 signed
// limbs of 27 bits in shared memory (radix 2^27, limbs below 2^27 + 2^9 in magnitude
// after a product, up to a few times that after sums), so additions and subtractions
// are limb-wise without carries, and a product is
//   1. columns: lane k sums the column sum_i x_i y_{k-i} in 64 bits (x read by
//      16-byte broadcasts, y by one word per lane and step);
//   2. one carry round: each column splits into three signed 27-bit digits, two of
//      which move up one and two lanes; limbs are bounded again, not canonical;
//   3. fold: the low 15 limbs t_k are replaced by t_k (2^(27 k) 2^-405 mod p), one
//      product with a constant column per lane, added to the high limbs. This is a
//      Montgomery reduction by 2^405 with one product instead of two, and leaves
//      about 2^27 p;
//   4. one more digit is taken off by adding m p with m = -V_0 mod 2^27 (p = 1 mod
//      2^27, so m needs no multiplication), and a carry round ends it.
// The result is x y 2^-432 mod p with |value| < 10 p. Every bound is in the text of
// the functions; the sums of products that the formulas need are formed in the
// columns, before step 2, so they cost one reduction.
//
// What bounds it: latency. About 15 multiply-adds, 20 shared-memory words, two
// shuffle rounds and one broadcast follow one another; an Edwards doubling (two
// levels of products, two barriers) takes 1157 cycles on GB300, a Weierstrass one 1299. The earlier form (12
// canonical 32-bit limbs, three column products and three ballot carry-lookaheads per
// product, separate levels for the sums) took 2277 cycles. The whole chain with its
// inversion: k_chain_w 614 -> 191 us (Weierstrass, n = 2^20, c = 16), 246 -> 100 us
// (Edwards + GLV, n = 13007, c = 10); k_window_horner_w 78 -> 36 and 38 -> 20 us.
//
// Curve forms. Edwards points are extended coordinates as in ed.cuh. Weierstrass
// points are homogeneous (X : Y : Z) with the formulas of Renes, Costello and Batina
// (2016) for a = 0, whose doubling has two levels of products where XYZZ has three.
// Their addition is exact except when P - Q has order 2, where all three
// coordinates vanish; add() notices that (see is_suspect) and takes the XYZZ law of
// ec.cuh on one thread for that addition. Both forms are projective, so a common
// power of two in all coordinates is allowed: coordinates read from memory (x 2^384
// mod p) enter as they are.
#pragma once
#include "ec.cuh"
#include "ed.cuh"

namespace wred {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kLimbs = 15, kBits = 27;
constexpr int kDigit = (1 << kBits) - 1, kHalf = 1 << (kBits - 1);

__device__ const static int kFold[kLimbs][16] = {
    {-58418647, 23545957, 38587369, -968839, -13364523, -12736573, -28016120, -59119190, -7407657, -32715674, -64567222, -18286210, -35111191, 23941973, 0, 0},
    {-56985136, 301609, 32869196, 56118023, -42770217, -51864758, -8704434, -30451620, -64361009, 53270663, -61650020, 47949316, -27465189, -5004327, 0, 0},
    {11910976, 43678160, 30336078, 40078203, -10799815, -64907888, -56703139, -1597972, 10950215, 6767123, -1184894, -39331836, 29998793, -7585463, 0, 0},
    {18054428, -11157696, -12574181, 21070998, 31960060, -36847982, 14077522, -43454190, -43192908, -19114416, -37194337, -3872858, -40366366, -10091849, 0, 0},
    {24019967, -295652, 20064568, -50460038, 55790877, -35251352, -37221549, -20016840, -12984730, -13681495, 37885138, -54959777, 51289601, -20981163, 0, 0},
    {49938007, 9864191, -1558610, -31960578, -2900981, -62847684, -35222782, -18003438, 64200921, -28464748, -38943410, 4552760, 50589886, -2710930, 0, 0},
    {6452379, -58589609, -46248947, -18038840, 61158890, -22787340, 55105516, -30219826, 22916144, -2973067, 3225453, -30816785, 48443489, -25675254, 0, 0},
    {61110579, 2782363, -20096795, -52357889, 57993537, 13344890, 17687811, -63266407, 49674763, -16912124, -12284388, -61130185, -39225787, -4080214, 0, 0},
    {9711462, 53770547, -63883506, -37033716, 38016550, -27469490, 45186141, 15046737, -12824504, -10103785, -26551163, -19466542, 54583640, -17752395, 0, 0},
    {42253102, 48508774, -10380702, -52852810, -53742511, -51441639, -58852989, -40314608, -17204553, 29924897, -32764749, 33868916, 55372329, -5779265, 0, 0},
    {13755432, -29050066, -13695816, -32154983, 31940574, -16301926, -41206073, 16010889, -2375565, -61317995, 62799059, 61490478, 43861418, -79315, 0, 0},
    {188780, -17701848, -62811024, 44639417, -64200861, 5227811, -31623864, 52789925, 24941693, 21064696, -67044339, 25458566, 24622506, 19269035, 0, 0},
    {-45862912, 188780, 4585144, 12686266, -23407279, -35200666, 38393219, 11474865, 35098397, -47192310, -22451081, -5475949, -57157822, 224, 0, 0},
    {-532, -10211328, -94317, -9693512, -37529123, 23347729, 24436378, -1791456, 63052212, -63093489, -39261606, -55568259, 22282005, 7709679, 0, 0},
    {-18350080, -532, 22931456, -94390, 9170288, 4401012, 5727111, -47837953, -19358532, 16665979, 43836029, -24924431, -56390796, 0, 0, 0},
};
// limbs of p, 32 p, and (all mod p) d 2^432 (Edwards d = k / 2), s 2^864, gamma 2^864, 2^864
__device__ const static int kP27[16] = {
    1, 18350080, 532, 111286272, 94389, 125047440, 129816715, 128490616,
    47837952, 19358532, 117551749, 90381698, 24924430, 56390796, 0, 0};
__device__ const static int k32P[16] = {
    32, 50331648, 17028, 71499776, 3020474, 109203968, 127603069, 85167902,
    54419486, 82602123, 3559588, 73642076, 126493141, 59675013, 13, 0};
__device__ const static int kD432[16] = {
    28739701, -62258772, -63384102, -61773890, 41397844, -52194151, -1628871, -33266492,
    -56125541, 23385514, -38434099, -52534755, 43501085, -23480652, 0, 0};
__device__ const static int kS864[16] = {
    940759, -8272637, 24297656, -61567514, -63830748, 20599720, -23338609, 60673254,
    -43884527, -52354120, 58673212, 46579060, -40990196, 940281, 0, 0};
__device__ const static int kGamma864[16] = {
    40552256, -15476456, 55348653, -16523777, -52366167, -6884464, -27342089, 10505923,
    2951248, -53863607, -48701043, -45718035, -47180760, -25412823, 0, 0};
__device__ const static int kOne864[16] = {
    -61265372, -29148207, -60229974, -24797738, -40753349, -39165604, 65494908, -50533739,
    58372182, 5850580, -25009488, -46161011, 41934807, -2966778, 0, 0};

// A slot holds one element: 16 zero words, 15 limbs and a zero, 16 zero words, so a
// lane may read limb k - i for every k < 32, i < 16.
constexpr int kSlotWords = 48;
enum : int { X = 0, Y = 1, Z = 2, T = 3,       // the accumulator
             kTmp = 4,                         // 4..9
             kQ = 10,                          // the operand, 10..13
             kRes = 14,                        // 14..16
             kC = 17,                          // a constant
             kRaw = 18,                        // 18..21
             kSlots = 22 };
// Shared words of a group: slots, one 16-word scratch per warp, flags.
constexpr int kSharedWords = kSlots * kSlotWords + 4 * 16 + 8;

struct Group {
    int* s;           // kSlots slots
    int* scr;         // this warp's scratch
    int* flags;       // 8 words
    int w, lane;      // warp of the group, lane
    int p;            // limb `lane` of p
    int c[kLimbs];    // limb `lane` of kFold[k]

    __device__ __forceinline__ int* limbs(int i) const { return s + kSlotWords * i + 16; }
    __device__ __forceinline__ int ld(int i) const { return limbs(i)[lane & 15]; }
    __device__ __forceinline__ void st(int i, int v) const {
        if (lane < kLimbs) limbs(i)[lane] = v;
    }
};

// mem: kSharedWords words of shared memory, 16-byte aligned; blocks of 128 threads.
__device__ __forceinline__ void init(Group& g, int* mem) {
    g.s = mem;
    g.w = threadIdx.x >> 5;
    g.lane = threadIdx.x & 31;
    g.scr = mem + kSlots * kSlotWords + 16 * g.w;
    g.flags = mem + kSlots * kSlotWords + 64;
    for (int i = threadIdx.x; i < kSharedWords; i += 128) mem[i] = 0;
    const int j = g.lane < 16 ? g.lane : 15;   // column 15 is zero
    g.p = kP27[j];
#pragma unroll
    for (int k = 0; k < kLimbs; ++k) g.c[k] = kFold[k][j];
    __syncthreads();
}

// Lane k: sum_i x_i y_{k-i} (zero from lane 29 on). |limbs| up to 2^29.5 each keep the
// 15 terms below 2^63.
__device__ __forceinline__ int64_t cols(const Group& g, int xs, int ys) {
    const int4* xv = reinterpret_cast<const int4*>(g.limbs(xs));
    const int* y = g.limbs(ys) + g.lane;
    const int4 a = xv[0], b = xv[1], c = xv[2], d = xv[3];
    int64_t s0 = (int64_t)a.x * y[0], s1 = (int64_t)a.y * y[-1];
    s0 += (int64_t)a.z * y[-2];
    s1 += (int64_t)a.w * y[-3];
    s0 += (int64_t)b.x * y[-4];
    s1 += (int64_t)b.y * y[-5];
    s0 += (int64_t)b.z * y[-6];
    s1 += (int64_t)b.w * y[-7];
    s0 += (int64_t)c.x * y[-8];
    s1 += (int64_t)c.y * y[-9];
    s0 += (int64_t)c.z * y[-10];
    s1 += (int64_t)c.w * y[-11];
    s0 += (int64_t)d.x * y[-12];
    s1 += (int64_t)d.y * y[-13];
    s0 += (int64_t)d.z * y[-14];
    return s0 + s1;
}

// Lane k: the column of x^2, by its symmetric pairs (floor(k/2) - d, ceil(k/2) + d).
__device__ __forceinline__ int64_t cols_sqr(const Group& g, int xs) {
    const int* x = g.limbs(xs);
    const int *lo = x + (g.lane >> 1), *hi = x + ((g.lane + 1) >> 1);
    const int64_t first = (int64_t)lo[0] * hi[0];
    int64_t s0 = 0, s1 = 0;
#pragma unroll
    for (int d = 1; d < 8; d += 2) {
        s0 += (int64_t)lo[-d] * hi[d];
        if (d + 1 < 8) s1 += (int64_t)lo[-d - 1] * hi[d + 1];
    }
    return ((s0 + s1) << 1) + ((g.lane & 1) ? first << 1 : first);
}

// The signed 27-bit digits of s: s = lo + 2^27 mid + 2^54 hi.
__device__ __forceinline__ int digit0(int64_t s) { return (int)((uint32_t)s << 5) >> 5; }
__device__ __forceinline__ int digit1(int64_t s) { return (int)((uint32_t)((s + kHalf) >> kBits) << 5) >> 5; }
__device__ __forceinline__ int digit2(int64_t s) { return (int)((s + kHalf + ((int64_t)kHalf << kBits)) >> (2 * kBits)); }

__device__ __forceinline__ int from_lane(int v, int src) { return __shfl_sync(kFull, v, src & 31); }

// sum of columns -> the reduced element, limb `lane` (lanes 15.. hold 0). Needs
// |columns| < 2^63 and the value below 2^(405 + 27) p. After the first carry round
// |t| <= 2^27 + 2^9; V adds 15 products below 2^53 and the high limb; with m p
// |V| < 2^58, so the last round leaves |limb| <= 2^27 + 2^4. The value is below
// 15 (2^27 + 2^9) (p / 2) / 2^27 + p / 2 + T / 2^432 < 10 p.
__device__ __forceinline__ int finish(const Group& g, int64_t s) {
    const int t = digit0(s) + from_lane(digit1(s), g.lane + 31) + from_lane(digit2(s), g.lane + 30);
    const int hi = from_lane(t, g.lane + kLimbs);
    __syncwarp();                                     // earlier readers of the scratch are done
    if (g.lane < kLimbs) g.scr[g.lane] = t;
    __syncwarp();
    const int4* tv = reinterpret_cast<const int4*>(g.scr);
    const int4 a = tv[0], b = tv[1], c = tv[2], d = tv[3];
    int64_t v0 = g.lane < kLimbs ? hi : 0;
    v0 += (int64_t)a.x * g.c[0];
    int64_t v1 = (int64_t)a.y * g.c[1];
    v0 += (int64_t)a.z * g.c[2];
    v1 += (int64_t)a.w * g.c[3];
    v0 += (int64_t)b.x * g.c[4];
    v1 += (int64_t)b.y * g.c[5];
    v0 += (int64_t)b.z * g.c[6];
    v1 += (int64_t)b.w * g.c[7];
    v0 += (int64_t)c.x * g.c[8];
    v1 += (int64_t)c.y * g.c[9];
    v0 += (int64_t)c.z * g.c[10];
    v1 += (int64_t)c.w * g.c[11];
    v0 += (int64_t)d.x * g.c[12];
    v1 += (int64_t)d.y * g.c[13];
    v0 += (int64_t)d.z * g.c[14];
    int64_t v = v0 + v1;
    const int m = -from_lane(digit0(v), 0);
    v += (int64_t)m * g.p;                            // column 0 is now a multiple of 2^27
    return from_lane(digit0(v), g.lane + 1) + digit1(v) + from_lane(digit2(v), g.lane + 31);
}

__device__ __forceinline__ int mul(const Group& g, int xs, int ys) { return finish(g, cols(g, xs, ys)); }

// Limb `lane` of the 12 packed words at w.
__device__ __forceinline__ int unpack(const uint32_t* w, int lane) {
    if (lane >= kLimbs) return 0;
    const int bit = kBits * lane, i = bit >> 5, sh = bit & 31;
    const uint32_t lo = w[i], hi = i + 1 < 12 ? w[i + 1] : 0u;
    return (int)(__funnelshift_r(lo, hi, sh) & (uint32_t)kDigit);
}

// c / R times (the integer in limbs l[0..14], |value| < 17 p, plus add0) mod p, in
// [0, 2p), on one thread: + 32 p, which keeps it positive and below 49 p < 2^384, carries,
// packing, and one Montgomery product by c (49 p c / R + p < 2 p).
__device__ __forceinline__ fq::fe to_fe_times(const int* l, int add0, const fq::fe& c) {
    uint32_t w[13];
#pragma unroll
    for (int k = 0; k < 13; ++k) w[k] = 0;
    int64_t carry = add0;
#pragma unroll
    for (int j = 0; j < kLimbs; ++j) {
        carry += (int64_t)l[j] + k32P[j];
        const uint64_t dig = (uint64_t)(carry & kDigit);
        carry >>= kBits;                              // arithmetic
        const int bit = kBits * j, i = bit >> 5, sh = bit & 31;
        const uint64_t v = dig << sh;
        w[i] |= (uint32_t)v;
        w[i + 1] |= (uint32_t)(v >> 32);
    }
    fq::fe a;
#pragma unroll
    for (int k = 0; k < 12; ++k) a.v[k] = w[k];
    fq::mul(a, a, c);
    return a;
}

// The integer itself mod p.
__device__ __forceinline__ fq::fe to_fe(const int* l, int add0) {
    fq::fe one;
    fq::set_one(one);
    return to_fe_times(l, add0, one);
}

// One thread: the limbs of a into slot i.
__device__ __forceinline__ void put_fe(const Group& g, int i, const fq::fe& a) {
    int* l = g.limbs(i);
    for (int j = 0; j < kLimbs; ++j) {
        const int bit = kBits * j, k = bit >> 5, sh = bit & 31;
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (int t = 0; t < 12; ++t) {
            if (t == k) lo = a.v[t];
            if (t == k + 1) hi = a.v[t];
        }
        l[j] = (int)(__funnelshift_r(lo, hi, sh) & (uint32_t)kDigit);
    }
}

// ---------------------------------------------------------------- inversion
//
// The inverse of z in [1, p) (12 words in shared memory) mod p, on one warp, by
// Bernstein and Yang's division steps ("Fast constant-time gcd computation and
// modular inversion", 2019) in the form that starts at delta = 1/2, whose bound on the steps
// is P. Wuille's (safegcd-bounds, 2021): with (delta, f, g) from
// (1/2, p, z), a step replaces (f, g) by (g, (g - f)/2) and delta by 1 - delta when
// delta > 0 and g is odd, and else (f, g) by (f, (g + (g mod 2) f)/2) and delta by
// 1 + delta. 27 steps depend on the low 27 bits only: they run on one register each
// (the same in every lane) and give a matrix (u v; q r) with rows of 1-norm at most
// 2^27, which is then applied to f, g and, mod p, to d, e with f = d z, g = e z. One
// division by 2^27 is one limb, so an application is two multiply-adds per lane and
// the carry round of a product. At most floor((45907 * 377 + 26313) / 19929) = 869
// steps bring g to 0, 33 rounds of 27; measured over random z: 27 to 29 rounds. Then f = +-1 and z^-1 = f d.
// About 20 us instead of 80 us for one thread's binary GCD (ec::inv).
constexpr int kInvRounds = 33;

// (a x + b y [+ m p]) / 2^27 per limb.
template <bool kMod>
__device__ __forceinline__ int shift_round(int lane, int p, int a, int x, int b, int y) {
    int64_t s = (int64_t)a * x + (int64_t)b * y;
    if (kMod) s += (int64_t)(-from_lane(digit0(s), 0)) * p;
    return from_lane(digit0(s), lane + 1) + digit1(s) + from_lane(digit2(s), lane + 31);
}

// p: limb `lane` of p. Limb `lane` of the inverse. A round replaces d and e, 0 and 1 at
// first, by (a d + b e + m p) / 2^27 with |a| + |b| <= 2^27 and |m| <= 2^26, so it adds at most
// p / 2 to the larger of their magnitudes: after the 33 rounds |value| <= 16.5 p + 1.
__device__ __forceinline__ int inverse(int lane, int p, const uint32_t* z) {
    int f = p, gg = unpack(z, lane), d = 0, e = lane == 0 ? 1 : 0;
    int delta2 = 1;                                    // 2 delta
    for (int round = 0; round < kInvRounds; ++round) {
        int fl = from_lane(f, 0), gl = from_lane(gg, 0);
        int u = 1, v = 0, q = 0, r = 1;
#pragma unroll 9
        for (int i = 0; i < kBits; ++i) {
            const bool odd = gl & 1, swap = odd && delta2 > 0;
            const int af = swap ? -fl : fl, au = swap ? -u : u, av = swap ? -v : v;
            fl = swap ? gl : fl;
            u = swap ? q : u;
            v = swap ? r : v;
            gl += odd ? af : 0;
            q += odd ? au : 0;
            r += odd ? av : 0;
            delta2 = swap ? 2 - delta2 : 2 + delta2;
            gl >>= 1;
            u <<= 1;
            v <<= 1;
        }
        const int f2 = shift_round<false>(lane, p, u, f, v, gg), g2 = shift_round<false>(lane, p, q, f, r, gg);
        const int d2 = shift_round<true>(lane, p, u, d, v, e), e2 = shift_round<true>(lane, p, q, d, r, e);
        f = f2;
        gg = g2;
        d = d2;
        e = e2;
        if (!__any_sync(kFull, gg != 0)) break;
    }
    return digit0(from_lane(f, 0)) < 0 ? -d : d;       // f = +-1
}

// a^-1 of lane `src`'s a (Montgomery form, nonzero mod p) in every lane, on one warp; mem:
// 28 words of shared memory of this warp's own.
constexpr int kInverseWords = 28;
__device__ __forceinline__ fq::fe inverse_fe(const fq::fe& a, int src, uint32_t* mem) {
    const int lane = threadIdx.x & 31;
    __syncwarp();                                      // earlier readers of mem are done
    if (lane == src) {
        fq::fe c;
        fq::canon(c, a);
        fq::store(mem, c);
    }
    __syncwarp();
    const int v = inverse(lane, kP27[lane < 16 ? lane : 15], mem);   // (a R)^-1
    int* limbs = reinterpret_cast<int*>(mem + 12);
    if (lane < 16) limbs[lane] = v;
    __syncwarp();
    fq::fe r3;
#pragma unroll
    for (int k = 0; k < fq::N; ++k) r3.v[k] = fq::kR3[k];
    return to_fe_times(limbs, 0, r3);                  // times R^2: a^-1 R
}

// ---------------------------------------------------------------- Edwards

struct Edwards {
    static __device__ __forceinline__ void set_inf(const Group& g) {   // (0 : 1 : 1 : 0)
        g.st(g.w, (g.w == Y || g.w == Z) && g.lane == 0 ? 1 : 0);
        __syncthreads();
    }

    // P = 2P (a = -1): E = 2 X Y, G = Y^2 - X^2, H = -(X^2 + Y^2), F = G - 2 Z^2,
    // each one sum of columns; X3 = E F, Y3 = G H, T3 = E H, Z3 = F G. T3 is needed
    // before an addition only (want_t). Columns stay below 4 * 15 * 2^54.1 < 2^60.1.
    static __device__ __forceinline__ void dbl(const Group& g, bool want_t) {
        int64_t s;
        if (g.w == 0) {
            s = cols(g, X, Y) << 1;
        } else {
            const int64_t xx = cols_sqr(g, X), yy = cols_sqr(g, Y);
            s = g.w == 2 ? -(xx + yy) : yy - xx;
            if (g.w == 3) s -= cols_sqr(g, Z) << 1;
        }
        g.st(kTmp + g.w, finish(g, s));                // E, G, H, F
        __syncthreads();
        if (g.w != 2 || want_t) {
            const int a = g.w == 1 ? kTmp + 1 : (g.w == 3 ? kTmp + 3 : kTmp);
            const int b = g.w == 0 ? kTmp + 3 : (g.w == 3 ? kTmp + 1 : kTmp + 2);
            g.st(g.w == 2 ? T : (g.w == 3 ? Z : g.w), finish(g, cols(g, a, b)));
        }
        __syncthreads();
    }

    // P += Q, Q in the operand slots as (X, Y, Z, d T): with e = X1 Y2 + Y1 X2,
    // h = Y1 Y2 + X1 X2, f = Z1 Z2 - T1 d T2, g = Z1 Z2 + T1 d T2 (the halves of the
    // E, H, F, G of ed.cuh), X3 = e f, Y3 = g h, T3 = e h, Z3 = f g. kStored: Q is a
    // stored point (x, y, Z = 1, u = 2 d x y) and e, h, Z1 Z2 are doubled instead.
    template <bool kStored>
    static __device__ __forceinline__ void add_op(const Group& g) {
        int64_t s;
        if (g.w < 2) {                                 // e, h
            s = cols(g, X, g.w == 0 ? kQ + Y : kQ + X) + cols(g, Y, g.w == 0 ? kQ + X : kQ + Y);
            if (kStored) s <<= 1;
        } else {                                       // f, g
            const int64_t c = cols(g, T, kQ + T);
            s = cols(g, Z, kQ + Z);
            if (kStored) s <<= 1;
            s += g.w == 2 ? -c : c;
        }
        g.st(kTmp + g.w, finish(g, s));
        __syncthreads();
        const int a = g.w == 1 ? kTmp + 3 : (g.w == 3 ? kTmp + 2 : kTmp);          // e, g, e, f
        const int b = g.w == 0 ? kTmp + 2 : (g.w == 3 ? kTmp + 3 : kTmp + 1);      // f, h, h, g
        g.st(g.w == 2 ? T : (g.w == 3 ? Z : g.w), finish(g, cols(g, a, b)));
        __syncthreads();
    }
    static __device__ __forceinline__ void add(const Group& g) { add_op<false>(g); }

    static __device__ __forceinline__ void load_const(const Group& g) {
        if (g.w == 0) g.st(kC, kD432[g.lane & 15]);
        __syncthreads();
    }

    // The operand slots from a packed point (X, Y, Z, T); all-zero words: the identity.
    static __device__ __forceinline__ void set_operand(const Group& g, int limb, bool zero_z) {
        const int v = zero_z ? ((g.w == Y || g.w == Z) && g.lane == 0 ? 1 : 0) : limb;
        g.st(g.w == T ? kRaw : kQ + g.w, v);
        __syncwarp();
        if (g.w == T) g.st(kQ + T, mul(g, kRaw, kC));  // d T
        __syncthreads();
    }

    // This warp's coordinate of the operand form (X, Y, Z, d T) of the accumulator.
    static __device__ __forceinline__ int as_operand(const Group& g) {
        return g.w == T ? mul(g, T, kC) : g.ld(g.w);
    }

    // The affine Weierstrass point of the accumulator in standard form (24 words), as
    // ed::to_weierstrass: with I = 1 / ((Z - Y) X) and r = (Z + Y) I, x = s X r - 1,
    // y = gamma Z r; the identity gives zeros.
    static __device__ __forceinline__ void store_affine(const Group& g, uint32_t* out) {
        if (g.w == 0) {
            g.st(kRaw, g.ld(Z) - g.ld(Y));
            __syncwarp();
            g.st(kTmp, mul(g, kRaw, X));
        } else if (g.w == 1) {
            g.st(kRaw + 1, g.ld(Z) + g.ld(Y));
        } else if (g.w == 2) {
            g.st(kRaw + 2, kS864[g.lane & 15]);
            __syncwarp();
            g.st(kTmp + 1, mul(g, kRaw + 2, X));
        } else {
            g.st(kRaw + 3, kGamma864[g.lane & 15]);
            __syncwarp();
            g.st(kTmp + 2, mul(g, kRaw + 3, Z));
        }
        __syncthreads();
        if (g.w == 0) {
            if (!invert_slot(g, kTmp, kQ)) {
                if (g.lane < 24) out[g.lane] = 0;
            }
            __syncwarp();
            g.st(kQ + 1, mul(g, kRaw + 1, kQ));        // r
        }
        __syncthreads();
        if (g.flags[0]) return;                        // block-uniform
        if (g.w < 2) {
            g.st(kRes + g.w, mul(g, kQ + 1, kTmp + 1 + g.w));
            __syncwarp();
            if (g.lane == 0) {
                fq::fe a = to_fe(g.limbs(kRes + g.w), g.w == 0 ? -1 : 0);
                fq::canon(a, a);
                fq::store(out + 12 * g.w, a);
            }
        }
    }

    // Warp 0: slot dst <- the inverse of slot src; false (and flags[0] set) when src = 0 mod p.
    static __device__ __forceinline__ bool invert_slot(const Group& g, int src, int dst) {
        uint32_t* z = reinterpret_cast<uint32_t*>(g.limbs(kRes));
        if (g.lane == 0) {
            fq::fe a = to_fe(g.limbs(src), 0);
            fq::canon(a, a);
            g.flags[0] = fq::is_zero_raw(a) ? 1 : 0;
            fq::store(z, a);
        }
        __syncwarp();
        const bool ok = g.flags[0] == 0;               // warp-uniform
        const int v = ok ? inverse(g.lane, g.p, z) : 0;
        g.st(dst, v);
        return ok;
    }
};

// ---------------------------------------------------------------- Weierstrass

struct Weierstrass {
    static __device__ __forceinline__ void set_inf(const Group& g) {   // (0 : 1 : 0)
        if (g.w < 3) g.st(g.w, g.w == Y && g.lane == 0 ? 1 : 0);
        __syncthreads();
    }

    // P = 2P on y^2 = x^3 + 1: U = Y^2 - 9 Z^2, V = Y^2 + 3 Z^2, X3 = 2 X Y U,
    // Y3 = U V + 24 (Y Z)^2, Z3 = 8 Y^2 (Y Z) with 8 Y^2 = 2 (U + 3 V). Columns: U below
    // 10 * 15 * 2^54.1 < 2^61.4, Y3 below 25 * 15 * 2^54.1 < 2^62.7. O and points of
    // order 2 need no case.
    static __device__ __forceinline__ void dbl(const Group& g, bool) {
        int64_t s;
        if (g.w == 0 || g.w == 2) {
            s = cols(g, Y, g.w == 0 ? X : Z);          // X Y, Y Z
        } else {
            const int64_t yy = cols_sqr(g, Y), zz = cols_sqr(g, Z);
            s = g.w == 1 ? yy - 9 * zz : yy + 3 * zz;  // U, V
        }
        g.st(kTmp + g.w, finish(g, s));                // XY, U, YZ, V
        __syncthreads();
        if (g.w == 0) {
            g.st(X, finish(g, cols(g, kTmp, kTmp + 1) << 1));
        } else if (g.w == 1) {
            g.st(Y, finish(g, cols(g, kTmp + 1, kTmp + 3) + 24 * cols_sqr(g, kTmp + 2)));
        } else if (g.w == 2) {
            g.st(kTmp + 4, g.ld(kTmp + 1) + 3 * g.ld(kTmp + 3));
            __syncwarp();
            g.st(Z, finish(g, cols(g, kTmp + 4, kTmp + 2) << 1));
        }
        __syncthreads();
    }

    // A coordinate of an exceptional sum is 0 mod p: q p with |q| < 16, so its limb 0
    // is q mod 2^27 (p = 1 mod 2^27). Any other value passes with probability 2^-22,
    // and passing only means the slow path.
    static __device__ __forceinline__ bool is_suspect(const Group& g, int limb) {
        const int q = digit0(from_lane(limb, 0));
        return q > -16 && q < 16;
    }

    // P += Q, Q in the operand slots (X, Y, Z): t3 = X1 Y2 + X2 Y1, a = Y1 Y2 - 3 Z1 Z2,
    // c = Y1 Y2 + 3 Z1 Z2, t4 = Y1 Z2 + Y2 Z1, q5 = 3 (X1 Z2 + X2 Z1), q0 = 3 X1 X2;
    // X3 = t3 a - t4 q5, Y3 = a c + q5 q0, Z3 = c t4 + q0 t3.
    static __device__ __forceinline__ void add(const Group& g) {
        int64_t s;
        if (g.w == 0 || g.w == 3) {                    // t3, t4
            const int o = g.w == 0 ? X : Z;
            s = cols(g, Y, kQ + o) + cols(g, o, kQ + Y);
        } else {                                       // a, c
            const int64_t zz = cols(g, Z, kQ + Z) * 3;
            s = cols(g, Y, kQ + Y) + (g.w == 1 ? -zz : zz);
        }
        g.st(kTmp + g.w, finish(g, s));
        if (g.w < 2) {                                 // q5, q0
            s = g.w == 0 ? cols(g, X, kQ + Z) + cols(g, Z, kQ + X) : cols(g, X, kQ + X);
            g.st(kTmp + 4 + g.w, finish(g, s * 3));
        }
        __syncthreads();
        if (g.w < 3) {
            // (t3, a, t4, q5), (a, c, q5, q0), (c, t4, q0, t3)
            const int b = g.w == 0 ? 1 : (g.w == 1 ? 2 : 3), c = g.w == 0 ? 3 : (g.w == 1 ? 4 : 5);
            const int d = g.w == 0 ? 4 : (g.w == 1 ? 5 : 0);
            const int64_t m = cols(g, kTmp + c, kTmp + d);
            const int r = finish(g, cols(g, kTmp + g.w, kTmp + b) + (g.w == 0 ? -m : m));
            g.st(kRes + g.w, r);
            const bool suspect = is_suspect(g, r);
            if (g.lane == 0) g.flags[g.w] = suspect ? 1 : 0;
        }
        __syncthreads();
        const bool slow = g.flags[0] && g.flags[1] && g.flags[2];   // block-uniform
        if (slow) {
            if (threadIdx.x == 0) add_thread(g);
        } else if (g.w < 3) {
            g.st(g.w, g.ld(kRes + g.w));
        }
        __syncthreads();
    }

    // The same sum by the XYZZ law on one thread.
    static __device__ __noinline__ void add_thread(const Group& g) {
        ec::xyzz P, Q;
        to_xyzz(g, X, P);
        to_xyzz(g, kQ, Q);
        ec::add(P, Q);
        fq::fe x, y, z;
        if (ec::is_inf(P)) {
            fq::set_zero(x);
            fq::set_one(y);
            fq::set_zero(z);
        } else {
            fq::mul(x, P.X, P.ZZZ);
            fq::mul(y, P.Y, P.ZZ);
            fq::mul(z, P.ZZ, P.ZZZ);
        }
        put_fe(g, X, x);
        put_fe(g, Y, y);
        put_fe(g, Z, z);
    }
    static __device__ __forceinline__ void to_xyzz(const Group& g, int base, ec::xyzz& P) {
        fq::fe x = to_fe(g.limbs(base), 0), y = to_fe(g.limbs(base + 1), 0), z = to_fe(g.limbs(base + 2), 0);
        if (fq::is_zero(z)) {
            ec::set_inf(P);
            return;
        }
        fq::mul(P.X, x, z);
        fq::mul(P.ZZ, z, z);
        fq::mul(P.Y, y, P.ZZ);
        fq::mul(P.ZZZ, P.ZZ, z);
    }

    static __device__ __forceinline__ void load_const(const Group&) {}

    // The operand slots from a packed XYZZ point: (X ZZZ : Y ZZ : ZZ ZZZ); ZZ = 0: (0 : 1 : 0).
    static __device__ __forceinline__ void set_operand(const Group& g, int limb, bool zero_z) {
        g.st(kRaw + g.w, limb);
        __syncthreads();
        if (g.w < 3) {
            const int a = g.w == 0 ? kRaw : (g.w == 1 ? kRaw + 1 : kRaw + 2);
            const int b = g.w == 1 ? kRaw + 2 : kRaw + 3;
            const int v = mul(g, a, b);
            g.st(kQ + g.w, zero_z ? (g.w == Y && g.lane == 0 ? 1 : 0) : v);
        }
        __syncthreads();
    }

    static __device__ __forceinline__ int as_operand(const Group& g) { return g.ld(g.w); }

    // The affine point of the accumulator in standard form (24 words); O gives zeros.
    static __device__ __forceinline__ void store_affine(const Group& g, uint32_t* out) {
        if (g.w == 1) g.st(kC, kOne864[g.lane & 15]);
        __syncthreads();
        if (g.w == 0) {
            if (!Edwards::invert_slot(g, Z, kQ)) {
                if (g.lane < 24) out[g.lane] = 0;
            }
        } else if (g.w < 3) {
            g.st(kTmp + g.w, mul(g, g.w - 1, kC));
        }
        __syncthreads();
        if (g.flags[0]) return;                        // block-uniform
        if (g.w == 1 || g.w == 2) {
            g.st(kRaw + g.w, mul(g, kTmp + g.w, kQ));
            __syncwarp();
            if (g.lane == 0) {
                fq::fe a = to_fe(g.limbs(kRaw + g.w), 0);
                fq::canon(a, a);
                fq::store(out + 12 * (g.w - 1), a);
            }
        }
    }
};

// A packed point in memory (four coordinates of 12 words): this warp's coordinate, read
// ahead of its use; zero_z says that coordinate 2 represents 0 (0 or p; all warps agree).
struct Packed {
    int limb;
    uint32_t z;   // word `lane` of coordinate 2
};
__device__ __forceinline__ Packed load_packed(const Group& g, const uint32_t* q) {
    Packed r;
    r.limb = unpack(q + 12 * g.w, g.lane);
    r.z = g.lane < 12 ? q[24 + g.lane] : 0u;
    return r;
}
__device__ __forceinline__ bool zero_z(const Group& g, const Packed& q) {
    const uint32_t p = g.lane < 12 ? fq::kP[g.lane] : 0u;
    return !__any_sync(kFull, q.z != 0u) || !__any_sync(kFull, q.z != p);
}

// A point in limb form (four coordinates of 16 words, operand form) in memory.
constexpr int kLimbPointWords = 64;
__device__ __forceinline__ int load_limbs(const Group& g, const int* q) {
    return g.lane < 16 ? q[16 * g.w + g.lane] : 0;
}

}  // namespace wred
