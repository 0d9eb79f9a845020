// Block fixed-point arithmetic for the FP64 solvers: 64-bit integers with one
// power-of-two exponent per vector and system, on the integer pipe.
//
// Why. On GB300 an FP64 warp-instruction takes an SM 19.3 clocks (measured:
// FMA, add and multiply alike), a 32 x 32 + 64 bit integer multiply-add 0.59
// and a 64-bit integer add 0.85, and the two pipes run side by side (six
// multiply-adds per FP64 FMA change nothing). The Krylov vectors of one system
// share a scale, so the exponent that FP64 keeps per entry can be kept once:
// an inner product or a matrix-vector product then is integer multiply-adds,
// 3 or 4 per term (2.4 clocks) where FP64 takes 19.3.
//
// Numbers. A vector y of a system is Y 2^e with Y int64, |Y| <= 2^57, and e
// one integer per vector. For products Y is split into two balanced digits,
// Y = hi 2^29 + lo, |hi| <= 2^28, |lo| <= 2^28. An entry carries 57 bits
// relative to the bound its vector was computed under, against FP64's 53
// relative to itself; every step's error is relative to the largest entry
// of its vector (block floating point), which is the measure the stopping
// test ||b - A x|| <= tau uses.
//   * Inner products keep all four partial products: exact up to a last
//     rounding at 2^-100 of the full scale.
//   * The matrix (Jacobi folded in, unit diagonal) is held as A 2^(60 - sigma)
//     where 2^sigma bounds its row sums; a product drops only lo lo, below
//     one unit of the result per stored entry.
//   * a + c y with a scalar c: c becomes a 58-bit integer relative to the
//     output's scale, three multiply-adds per term.
// A result's exponent is fixed before it is computed, from bounds of its
// terms: the measured bit lengths of the vectors involved (they ride on the
// reductions) and the scalars' exponents. No entry can overflow.
//
// What bounds it now: latency (fixed-latency dependences and instruction
// fetch; 12 warps of 168 registers on an SM, 42 % of the issue slots used, FP64
// unit 4 %). Measured, start (FP64 pipe 94 % of its rate) -> now:
//   65,536 systems, n = 144, 5-point, CSR, 16 lanes   12.03 -> 5.79 ms
//   131,072 systems, n = 22, dense, 8 lanes            3.58 -> 1.46 ms
//   16,384 systems, n = 144, 43 values a row          12.95 -> 8.6 ms
//   4,096 systems, n = 1,024, 9-point, 4 warps        14.63 -> 6.5 ms
// The iteration counts of the first batch are the same (mean 23.135).
//
// What is left to the FP64 code: a system whose numbers do not fit (a zero or
// missing diagonal entry, row sums of the scaled matrix of 31 or more, non-finite
// entries, a matrix beyond FP32's range, a right-hand side or guess scaled beyond
// 2^+-400, equations of scales too far apart or weak diagonal dominance, see
// folded_setup), one that breaks down, stagnates or misses the tolerance once x is
// rounded to FP64, and all without Jacobi. It is staged again where its values have been
// overwritten; nothing has been written for it by then. Such systems pay for both:
// batches of n = 144 of them alone take 4 to 12 % longer than FP64 did, and every other
// one of 16,384, in the same warps, 5.8 ms where FP64 took 3.3 for all.
#pragma once

#include "bbs_solvers.cuh"

namespace bbs {
namespace fx {

constexpr int kNone = -1000000;  // exponent of a vector that is zero
constexpr float kRowSumMax = 31.0f;
// What a system must be like to be solved here, and what became of it.
constexpr float kExcess = 0x1p-7f;    // BiCGSTAB: least diagonal excess of a row, (|a_ii| - sum of the others) / |a_ii|
constexpr float kExcessCg = 0x1p-9f;  // CG
constexpr float kRowScale = 0x1p-12f; // smallest row scale against the largest
constexpr int kRowScaleBits = 12;
constexpr int kDiagonalBits = 24;     // CG: spread of the diagonal
// Statuses that end a solve here; of a system that stops in another way nothing is
// written.
constexpr int kStagnated = -2;
__device__ __forceinline__ bool accepted(int status) { return status == ST_CONVERGED || status == ST_MAX_ITER; }
enum Fit { kUnfit, kDone, kLeft };    // not begun (the staged values are intact), solved, given up (they are not)
constexpr int kMaxWarps = 16;  // warps of a team whose partial sums fit the reduction area

struct Dig {
    int hi, lo;
};

// p, which points into the block's dynamic shared memory, as a pointer that
// the compiler sees to be one (32-bit addresses with immediate offsets).
template <typename T>
__device__ __forceinline__ T* in_shared(const void* p) {
#ifdef __CUDA_ARCH__
    extern __shared__ __align__(16) unsigned char raw[];
    const unsigned base = static_cast<unsigned>(__cvta_generic_to_shared(raw));
    return reinterpret_cast<T*>(raw + (static_cast<unsigned>(__cvta_generic_to_shared(p)) - base));
#else
    return reinterpret_cast<T*>(const_cast<void*>(p));
#endif
}

// c + a b, one multiply-add. The product is written as PTX: 65,536 systems of n =
// 144 take 6.19 ms with it and 10.0 ms with c + (long long)a * b; CG on 30,001 of n
// = 143 2.26 and 3.35 ms.
__device__ __forceinline__ long long wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return c + r;
#else
    return c + (long long)a * b;
#endif
}
__device__ __forceinline__ Dig split(long long y) {
    Dig d;
    d.hi = (int)((y + (1ll << 28)) >> 29);
    d.lo = (int)((unsigned)y << 3) >> 3;
    return d;
}
__device__ __forceinline__ long long join(Dig d) { return wide(d.hi, 1 << 29, (long long)d.lo); }
__device__ __forceinline__ Dig dig(int2 v) { return Dig{v.x, v.y}; }
__device__ __forceinline__ int2 pack(Dig d) { return make_int2(d.hi, d.lo); }

// c 2^s for c = 0 or c and the result in the normal range.
__device__ __forceinline__ double scale2(double c, int s) {
    const int hi = __double2hiint(c);
    return __hiloint2double((hi & 0x7ff00000) ? (int)((unsigned)hi + ((unsigned)s << 20)) : 0, __double2loint(c));
}
// y >> d for any d >= 0 (63 and more: the sign)
__device__ __forceinline__ long long shr(long long y, int d) { return y >> min((unsigned)d, 63u); }
// Every y >> d, d >= 0 (two funnel shifts a row; 32 places and more are rare:
// one vector has been swamped by another).
template <int R, class G>
__device__ __forceinline__ void shr_rows(long long (&y)[R], int d, const G& g) {
    if (g.any(d > 31)) {
        const int far = d > 31 ? min(d, 62) - 31 : 0;
#pragma unroll
        for (int q = 0; q < R; ++q) y[q] >>= far;
        d = min(d, 31);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int hi = (int)(y[q] >> 32);
        y[q] = ((long long)(hi >> d) << 32) | __funnelshift_r((unsigned)y[q], (unsigned)hi, d);
    }
}
// y << k, 0 <= k <= 31
__device__ __forceinline__ long long shl31(long long y, int k) {
    const unsigned lo = (unsigned)y;
    return ((long long)(int)__funnelshift_l(lo, (unsigned)(y >> 32), k) << 32) | (unsigned)(lo << k);
}

// Shifts a residual of `bits` bits (44: or fewer, then its length is taken first)
// up to 56, its exponent e following.
template <int R, class G>
__device__ __forceinline__ void fill_up(long long (&y)[R], int& e, int& bits, G& g) {
    int k = max(0, 56 - bits);
    if (g.any(bits <= 44)) {  // rare: it has fallen by 2^12 and more since it was last shifted
        unsigned long long o = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) o |= (unsigned long long)(y[q] ^ (y[q] >> 63));
        const int length = g.max_int(64 - __clzll((long long)o));
        if (bits <= 44) k = 56 - length;
        const int far = max(0, k - 31);
#pragma unroll
        for (int q = 0; q < R; ++q) y[q] = (long long)((unsigned long long)y[q] << far);
        k -= far;
        e -= far;
        if (bits <= 44) bits = 56 - k;  // (the others' k is theirs: no group sees its neighbours)
    }
    e -= k;
    bits += k;
#pragma unroll
    for (int q = 0; q < R; ++q) y[q] = shl31(y[q], k);
}

// Sum of c y terms: hh in units of the result, m in units of 2^-29.
struct Sum {
    long long hh, m;
    __device__ __forceinline__ void add(Dig c, Dig y) {
        hh = wide(c.hi, y.hi, hh);
        m = wide(c.hi, y.lo, m);
        m = wide(c.lo, y.hi, m);
    }
    __device__ __forceinline__ long long value() const { return hh + (m >> 29); }
};

// Inner product of the caller's rows: all four partial products.
struct Dot {
    long long hh, m, ll;
    __device__ __forceinline__ void clear() { hh = m = ll = 0; }
    __device__ __forceinline__ void add(Dig a, Dig b) {
        hh = wide(a.hi, b.hi, hh);
        m = wide(a.hi, b.lo, m);
        m = wide(a.lo, b.hi, m);
        ll = wide(a.lo, b.lo, ll);
    }
    __device__ __forceinline__ void square(Dig a) {
        hh = wide(a.hi, a.hi, hh);
        m = wide(a.hi, 2 * a.lo, m);
        ll = wide(a.lo, a.lo, ll);
    }
};

// Inner product of R rows of vectors whose high digits reach 2^30 (results of
// spmv_fixed): hh is carried out every four rows.
template <int R>
__device__ __forceinline__ Dot dot_wide(const Dig (&a)[R], long long& carry) {
    Dot d;
    d.clear();
    carry = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        d.square(a[q]);
        if ((q & 3) == 3 && q + 1 < R) {
            carry += d.hh >> 10;
            d.hh &= 1023;
        }
    }
    return d;
}

// A partial sum on its way through the reduction: hi 2^54 + lo in units of 2^14,
// 0 <= lo < 2^54. Sums over 2048 rows of products of 2^118 stay below 2^63 in
// hi, and 512 lanes' lo below 2^63. The bits below 2^14 are dropped: 2^-100 of
// the full scale, so a vector whose entries have cancelled down to 2^40 units
// still has a norm of 53 bits. (At 2^47, with 21 bits in lo, one of 2^32 units had
// 17 bits, and one of 2^23 the norm 0: omega = 0 then stopped systems that FP64
// solves, 28 of 300 with the matrix tridiag(-1, 2, -1), n = 128.)
struct Part {
    long long hi, lo;
};
__device__ __forceinline__ Part part(const Dot& d, long long carry = 0) {
    constexpr long long kLow = (1 << 29) - 1;
    const long long m = d.m + (d.ll >> 29);
    const long long h = d.hh + (m >> 29);
    Part p;
    p.hi = (h >> 10) + carry;
    p.lo = (h & 1023) << 44 | (m & kLow) << 15 | (d.ll & kLow) >> 14;
    return p;
}
// A scalar m 2^e with 2^61 <= |m| < 2^62 (zero: m = 0, e = kNone). The
// iteration's scalars stay on the integer pipe too: an FP64 operation occupies
// its scheduler's FP64 unit for 64 clocks and more, and a division is a chain
// of eight.
struct Sc {
    long long m;
    int e;
};
__device__ __forceinline__ Sc normal(long long v, int e) {
    const int z = __clzll(v ^ (v >> 63)) - 2;
    Sc s;
    s.m = (long long)((unsigned long long)v << z);
    s.e = v == 0 ? kNone : e - z;
    return s;
}
// The sum of vectors whose exponents add up to e.
__device__ __forceinline__ Sc value(Part p, int e) {
    const long long hi = p.hi + (p.lo >> 54);
    const long long lo = p.lo & ((1ll << 54) - 1);
    const int z = min(__clzll(hi ^ (hi >> 63)) - 2, 54);
    const long long v = (long long)((unsigned long long)hi << z) + (lo >> (54 - z));
    return normal(v, 68 - z + e);
}
__device__ __forceinline__ Sc one() { return Sc{1ll << 61, -61}; }
// c, exactly (zero below the normal range; infinities come out as 2^1024 and more)
__device__ __forceinline__ Sc unpack(double c) {
    const int hi = __double2hiint(c), E = (hi >> 20) & 0x7ff;
    const long long m = ((long long)((hi & 0xfffff) | 0x100000) << 41) | ((long long)(unsigned)__double2loint(c) << 9);
    return E == 0 ? Sc{0, kNone} : Sc{hi < 0 ? -m : m, E - 1084};
}
// y 2^-d rounded, 1 <= d (0 from 63 on)
__device__ __forceinline__ long long round_shr(long long y, int d) {
    return d > 62 ? 0 : (y + (1ll << (d - 1))) >> d;
}
// c 2^s rounded to an integer below 2^61.
__device__ __forceinline__ long long to_int(double c, int s) {
    const Sc u = unpack(c);
    return round_shr(u.m, -(u.e + s));
}
__device__ __forceinline__ double to_double(Sc a) {
    const int E = a.e + 62 + 1022;  // biased exponent of the result, rounding aside
    if (a.m == 0 || E <= 1) return 0.0;
    const double v = __ll2double_rn(a.m);
    return E >= 2046 ? v * __longlong_as_double(0x7ff0000000000000LL) : scale2(v, a.e);
}
__device__ __forceinline__ Sc neg(Sc a) { return Sc{-a.m, a.e}; }
// |c| < (1 - 2^-29) 2^ex(c)
__device__ __forceinline__ int ex(Sc c) {
    const int h = (int)(c.m >> 32);
    return c.e + 62 + ((h ^ (h >> 31)) >= 0x3ffffffe ? 1 : 0);
}
// In FP64's range, as the FP64 solvers test it: overflow is not finite,
// underflow is zero.
__device__ __forceinline__ bool finite(Sc a) { return a.e < 1024 - 62; }
__device__ __forceinline__ bool zero(Sc a) { return a.e < -1074 - 62; }
// a <= b, both >= 0
__device__ __forceinline__ bool le(Sc a, Sc b) { return a.e < b.e || (a.e == b.e && a.m <= b.m); }

// High 62 bits of a product, rounded (the two low halves' product, below one unit,
// is left out).
__device__ __forceinline__ long long mul62(long long a, long long b) {
    const int ah = (int)(a >> 31), bh = (int)(b >> 31);
    const int al = (int)((unsigned)a & 0x7fffffffu), bl = (int)((unsigned)b & 0x7fffffffu);
    return wide(ah, bh, wide(ah, bl, wide(al, bh, 1 << 30)) >> 31);
}
__device__ __forceinline__ Sc mul(Sc a, Sc b) {
    const long long r = mul62(a.m, b.m);
    const bool small = ((r ^ (r >> 63)) >> 61) == 0;  // below 2^61
    return Sc{small ? r + r : r, a.m == 0 || b.m == 0 ? kNone : a.e + b.e + 62 - (small ? 1 : 0)};
}
// 1 / a: an FP32 reciprocal and two Newton steps in fixed point. With
// x = |m| / 2^62 in [1/2, 1), y 2^61 ~ 1 / x: y += y (1 - x y) takes the 23 bits
// of FP32 to 44 and to 60. (1 / 0: some finite number.)
__device__ __forceinline__ Sc rcp(Sc a) {
    const long long x = a.m < 0 ? -a.m : a.m;
    const int xh = (int)(x >> 31);  // x 2^31
    // (FP32 rounding may reach 2: kept below)
    const float f = fminf(__frcp_rn((float)xh * 4.656612873077393e-10f), 1.9999998f);
    long long y = (long long)(int)(f * 1073741824.0f) << 31;
    {
        const long long d = (1ll << 61) - mul62(x, y);  // 2^61 (1 - x y), below 2^40
        const int dh = (int)(d >> 10);
        y += wide((int)(y >> 31), dh, 0) >> 20;
    }
    {
        const long long d = (1ll << 61) - mul62(x, y);  // below 2^20
        y += wide((int)(y >> 31), (int)d, 0) >> 30;
    }
    const bool two = y >= (1ll << 62);  // |m| = 2^61 exactly
    if (two) y = (1ll << 62) - 1;
    return Sc{a.m < 0 ? -y : y, -a.e - 123};
}
// The multiplier of a term c y (y at exponent ey) in a result at exponent
// eo >= ey + ex(c) - 2: c 2^(ey - eo), below 4 (1 - 2^-29) so that the high
// digit fits 32 bits, in units of 2^-58.
__device__ __forceinline__ Dig coef(Sc c, int ey, int eo) { return split(shr(c.m, eo - ey - c.e - 58)); }

// The high digits of a vector, or-ed with their signs taken off, give its bit
// length; two vectors' masks travel as the two halves of a word, 16 bits each
// (a vector below 2^44 counts as one of 44 bits).
__device__ __forceinline__ unsigned mag(int hi) { return (unsigned)(hi ^ (hi >> 31)); }
__device__ __forceinline__ unsigned masks(unsigned a, unsigned b) { return (a >> 15) << 16 | (b >> 15); }
__device__ __forceinline__ int bits_first(unsigned o) { return max(44, 60 - __clz((int)(o & 0xffff0000u))); }
__device__ __forceinline__ int bits_second(unsigned o) { return max(44, 60 - __clz((int)(o << 16))); }

// --------------------------------------------------- the lanes of a system

// Sums of ND = 1, 2 or 3 partial sums over each aligned group of L lanes,
// transposed as group_sum does it: the first levels exchange half of the
// values. Lane l ends up with the sum of index which<L, ND>(l).
__device__ __forceinline__ Part plus(Part a, Part b, int m) {
    return Part{a.hi + shfl_xor(b.hi, m), a.lo + shfl_xor(b.lo, m)};
}
template <int L, int ND>
__device__ __forceinline__ int which(int lane) {
    if constexpr (ND == 1) return 0;
    if constexpr (ND == 2) return lane & (L / 2) ? 1 : 0;
    return (lane & (L / 2) ? 2 : 0) + (lane & (L / 4) ? 1 : 0);
}
template <int L, int ND>
__device__ __forceinline__ int home(int j) {  // a lane that ends up with sum j
    return ND == 1 ? 0 : ND == 2 ? j * (L / 2) : (j & 2) / 2 * (L / 2) + (j & 1) * (L / 4);
}
template <int L, int ND>
__device__ __forceinline__ Part lane_sums(const Part (&p)[ND], int lane) {
    static_assert(ND >= 1 && ND <= 3, "1 to 3 sums");
    Part k = p[0];
    int top = L / 2;
    if constexpr (ND == 2) {
        const bool b = lane & (L / 2);
        k = plus(b ? p[1] : p[0], b ? p[0] : p[1], L / 2);
        top = L / 4;
    } else if constexpr (ND == 3) {
        const bool b = lane & (L / 2), c = lane & (L / 4);
        const Part zero{0, 0};
        const Part k0 = plus(b ? p[2] : p[0], b ? p[0] : p[2], L / 2);
        const Part k1 = plus(b ? zero : p[1], b ? p[1] : zero, L / 2);
        k = plus(c ? k1 : k0, c ? k0 : k1, L / 4);
        top = L / 8;
    }
#pragma unroll
    for (int m = top; m; m >>= 1) k = plus(k, k, m);
    return k;
}

// An aligned group of L lanes of a warp that runs in lockstep with the
// warp's other groups.
template <int L>
struct Lanes {
    static constexpr int kLanes = L;
    int lane;
    __device__ __forceinline__ void sync() const { __syncwarp(); }
    __device__ __forceinline__ bool any(bool p) const { return __any_sync(kFull, p); }
    // Whether any warp of the block goes on: keeps the block's warps, one on
    // each scheduler, within an iteration of each other.
    __device__ __forceinline__ bool live(bool p) const {
        return blockDim.x == 32 ? __any_sync(kFull, p) : __syncthreads_or(p) != 0;
    }
    __device__ __forceinline__ int max_int(int v) const {
#pragma unroll
        for (int s = L / 2; s; s >>= 1) v = max(v, shfl_xor(v, s));
        return v;
    }
    // out[j] = the sum of p[j], its vectors' exponents adding up to e[j]; o or-ed
    template <int ND, typename O>
    __device__ __forceinline__ void sums(const Part (&p)[ND], const int (&e)[ND], Sc (&out)[ND], O& o) {
#pragma unroll
        for (int s = L / 2; s; s >>= 1) o |= shfl_xor(o, s);
        const Part k = lane_sums<L, ND>(p, lane);
        if constexpr (ND == 1) {
            out[0] = value(k, e[0]);
        } else {
            const int w = which<L, ND>(lane);
            int we = e[0];
#pragma unroll
            for (int j = 1; j < ND; ++j) we = w == j ? e[j] : we;
            const Sc d = value(k, we);
            const int base = lane & ~(L - 1);
#pragma unroll
            for (int j = 0; j < ND; ++j) out[j] = Sc{shfl(d.m, base + home<L, ND>(j)), shfl(d.e, base + home<L, ND>(j))};
        }
    }
};

// A team of whole warps (one system): warp sums by shuffles, across warps
// through the reduction area (two halves in turn, one barrier each).
struct Warps {
    static constexpr int kLanes = 0;
    Team tm;
    unsigned char* red;
    int parity;
    __device__ __forceinline__ void sync() const { tm.sync(); }
    __device__ __forceinline__ bool any(bool p) const { return p; }
    __device__ __forceinline__ bool live(bool p) const { return p; }
    __device__ __forceinline__ unsigned char* half() {
        unsigned char* r = red + parity * 1024;
        parity ^= 1;
        return r;
    }
    __device__ __forceinline__ static unsigned or_all(unsigned o) { return __reduce_or_sync(kFull, o); }
    __device__ __forceinline__ static unsigned long long or_all(unsigned long long o) {
        return (unsigned long long)or_all((unsigned)(o >> 32)) << 32 | or_all((unsigned)o);
    }
    __device__ __forceinline__ int max_int(int v) {
        v = __reduce_max_sync(kFull, v);
        if (tm.nwarps == 1) return v;
        int* r = reinterpret_cast<int*>(half());
        if (tm.lane == 0) r[tm.warp] = v;
        tm.sync();
        for (int w = 0; w < tm.nwarps; ++w) v = max(v, r[w]);
        return v;
    }
    template <int ND, typename O>
    __device__ __forceinline__ void sums(const Part (&p)[ND], const int (&e)[ND], Sc (&out)[ND], O& o) {
        o = or_all(o);
        const Part k = lane_sums<32, ND>(p, tm.lane);
        const int w = which<32, ND>(tm.lane);
        if (tm.nwarps == 1) {
            int we = e[0];
#pragma unroll
            for (int j = 1; j < ND; ++j) we = w == j ? e[j] : we;
            const Sc d = value(k, we);
#pragma unroll
            for (int j = 0; j < ND; ++j) out[j] = Sc{shfl(d.m, home<32, ND>(j)), shfl(d.e, home<32, ND>(j))};
            return;
        }
        // slot of a warp: hi[3] | lo[3] | mask (4 or 8 bytes), 64 bytes in all
        unsigned char* r = half();
        if (w < ND && tm.lane == home<32, ND>(w)) {
            unsigned char* slot = r + tm.warp * 64;
            reinterpret_cast<long long*>(slot)[w] = k.hi;
            reinterpret_cast<long long*>(slot + 24)[w] = k.lo;
            if (w == 0) *reinterpret_cast<O*>(slot + 48) = o;
        }
        tm.sync();
        Part t[ND];
#pragma unroll
        for (int j = 0; j < ND; ++j) t[j] = Part{0, 0};
        for (int v = 0; v < tm.nwarps; ++v) {
            const unsigned char* slot = r + v * 64;
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                t[j].hi += reinterpret_cast<const long long*>(slot)[j];
                t[j].lo += reinterpret_cast<const long long*>(slot + 24)[j];
            }
            o |= *reinterpret_cast<const O*>(slot + 48);
        }
#pragma unroll
        for (int j = 0; j < ND; ++j) out[j] = value(t[j], e[j]);
    }
};

// ------------------------------------------------------------ the matrix

// f(position, column) for the stored entries of a row in the staged layout
// (column -1: padding).
template <int SF, class F>
__device__ __forceinline__ void each_entry(const Mat<double>& S, int row, F f) {
    if constexpr (SF == FMT_CSR) {
        const int e1 = ldg(S.row_ptrs + row + 1);
#pragma unroll 2
        for (int e = ldg(S.row_ptrs + row); e < e1; ++e) f(e, ldg(S.cols + e));
    } else if constexpr (SF == FMT_ELL) {
#pragma unroll 2
        for (int j = 0; j < S.k; ++j) f(j * S.n + row, ldg(S.cols + (size_t)j * S.n + row));
    } else {
#pragma unroll 2
        for (int j = 0; j < S.n; ++j) f(row * S.n + j, j);
    }
}

// Sum of |c| |y| to the high digits, as `Sum` for spmv_sums.
struct Abs {
    long long hh;
    __device__ __forceinline__ void add(Dig c, Dig y) { hh = wide(abs(c.hi), abs(y.hi), hh); }
};
__device__ __forceinline__ void begin(Sum& s, int round) { s = Sum{0, round}; }
__device__ __forceinline__ void begin(Abs& s, int) { s = Abs{0}; }

// Dense digits are kept by rows as the values are, but by columns where rows
// of n 8-byte words put 16 or 32 lanes on the same banks (16,384 systems of n =
// 144: 42.5 ms by rows, 18.1 ms by columns; n = 54: 1.99 ms by rows, 2.30 ms by
// columns, whose digits are made from values read again from global memory).
__device__ __forceinline__ bool by_columns(int n) { return (n & 7) == 0; }

template <int R>
__device__ __forceinline__ void carry(Abs (&)[R]) {}
template <int R>
__device__ __forceinline__ void carry(Sum (&s)[R]) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
        s[q].hh += s[q].m >> 29;
        s[q].m &= (1 << 29) - 1;
    }
}

// A Y for the caller's rows: `a` the staged digits, `y` the vector's digits in
// shared memory. hh comes in units of y's exponent plus sigma - 2, below 2^59
// (sum |A hi| |Y hi| <= 2^31 2^28), m as the 29 bits below it, rounded by
// `round`. Between carries m holds kTerms terms of 2^57 (of 2^59 where |Y| goes
// to 2^59, and hh to 2^61). The slots are the outer loop: R rows' loads are in
// flight at once, and the loop's code stays within the instruction cache (all
// rows' slots unrolled took 5 times the code and ran 8 times slower).
template <int SF, int kTerms, class T, int R>
__device__ __forceinline__ void spmv_sums(const Mat<double>& S, const int2* __restrict__ a,
                                          const int2* __restrict__ y, T (&s)[R], int round, const Team& tm) {
#pragma unroll
    for (int q = 0; q < R; ++q) begin(s[q], round);
    // Only the last row may lie past the end: such a lane repeats its first row
    // in its place (row 0 if it has none) and drops the result, so that the
    // loops need no branch.
    const bool last = tm.row(R - 1) < S.n;
    const int rl = last ? tm.nt * (R - 1) : 0;
    const int first = R > 1 || last ? tm.tid : 0;
    const auto off = [&](int q) { return q + 1 < R ? q * tm.nt : rl; };
    if constexpr (SF == FMT_CSR) {
        int e[R], len[R], most = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int row = tm.row(q);
            const bool ok = q + 1 < R || last;
            e[q] = ok ? ldg(S.row_ptrs + row) : 0;
            len[q] = ok ? ldg(S.row_ptrs + row + 1) - e[q] : 0;
            most = max(most, len[q]);
        }
        most = __reduce_max_sync(kFull, most);
#pragma unroll 1
        for (int j0 = 0; j0 < most; j0 += kTerms) {
            const int j1 = min(most, j0 + kTerms);
#pragma unroll 1
            for (int j = j0; j < j1; ++j)
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (j < len[q]) s[q].add(dig(a[e[q] + j]), dig(y[ldg(S.cols + e[q] + j)]));
            carry(s);
        }
    } else if constexpr (SF == FMT_ELL) {
        const int32_t* c = S.cols + first;
        const int2* ar = a + first;
#pragma unroll 1
        for (int j0 = 0; j0 < S.k; j0 += kTerms) {
            const int j1 = min(S.k, j0 + kTerms);
#pragma unroll 2
            for (int j = j0; j < j1; ++j) {
#pragma unroll
                for (int q = 0; q < R; ++q)  // (padding: zero digits)
                    s[q].add(dig(ar[off(q)]), dig(y[max(ldg(c + off(q)), 0)]));
                c += S.n;
                ar += S.n;
            }
            carry(s);
        }
    } else {
        const int rs = by_columns(S.n) ? 1 : S.n, cs = by_columns(S.n) ? S.n : 1;
        const int2* ar = a + first * rs;
#pragma unroll 1
        for (int j0 = 0; j0 < S.n; j0 += kTerms) {
            const int j1 = min(S.n, j0 + kTerms);
#pragma unroll 2
            for (int j = j0; j < j1; ++j) {
                const Dig yj = dig(y[j]);
#pragma unroll
                for (int q = 0; q < R; ++q) s[q].add(dig(ar[off(q) * rs]), yj);
                ar += cs;
            }
            carry(s);
        }
    }
#pragma unroll
    for (int q = 0; q < R; ++q)
        if (q + 1 == R && !last) begin(s[q], 0);
}

// Their digits, rounded to units of y's exponent plus sigma - 2.
template <int SF, int R>
__device__ __forceinline__ void spmv_fixed(const Mat<double>& S, const int2* __restrict__ a,
                                           const int2* __restrict__ y, Dig (&v)[R], const Team& tm) {
    Sum s[R];
    spmv_sums<SF, 64>(S, a, y, s, 1 << 28, tm);
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = split(s[q].hh);
}

// A residual b - A x, of which most leading bits have cancelled: shifts it so
// that its largest entry has 56 bits (its exponent e follows), and returns its
// squared norm.
template <int R, class G>
__device__ __forceinline__ Sc norm2_full(long long (&y)[R], int& e, G& g) {
    unsigned long long o = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) o |= (unsigned long long)(y[q] ^ (y[q] >> 63));
    const int k = 56 - g.max_int(64 - __clzll((long long)o));
    const int up = max(k, 0), down = max(-k, 0);
    Dot d;
    d.clear();
#pragma unroll
    for (int q = 0; q < R; ++q) {
        y[q] = (long long)((unsigned long long)y[q] << up) >> down;
        d.square(split(y[q]));
    }
    e -= k;
    const Part pt[1] = {part(d)};
    const int pe[1] = {2 * e};
    Sc r[1];
    unsigned none = 0;
    g.sums(pt, pe, r, none);
    return r[0];
}

// ||b - A x||^2 (x through buf). A group with `take` set keeps b - A x in r,
// and x with its units made finer.
template <int SF, int R, class G>
__device__ __forceinline__ Sc true_residual(const Mat<double>& S, const int2* as, int2* buf, const SysIO& io, int sigma,
                                            long long (&X)[R], int& eX, int& bX, long long (&Rv)[R], int& eR, int& bR,
                                            bool take, G& g, const Team& tm, int* e_digits = nullptr) {
    const int n = io.n;
    // x with 59 bits: shifted up exactly where it holds fewer (a guess far above
    // the solution has left it coarse units), else rounded for the product
    unsigned long long xo = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) xo |= (unsigned long long)(X[q] ^ (X[q] >> 63));
    const int k = 59 - g.max_int(64 - __clzll((long long)xo));
    const int up = k > 0 && k < 59 ? k : 0, dx = max(-k, 0), ex4 = eX - up + dx;
    if (e_digits != nullptr) *e_digits = ex4;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = tm.row(q);
        const long long y = (long long)((unsigned long long)X[q] << up);
        if (row < n) buf[row] = pack(split((y + ((1ll << dx) >> 1)) >> dx));
        if (take) X[q] = y;
    }
    if (take) {  // (a system's bits do not depend on the warp's others)
        eX -= up;
        bX = 59 - min(k, 0);
    }
    g.sync();
    Sum t[R];
    spmv_sums<SF, 16>(S, as, buf, t, 1 << 27, tm);
    int eb = 0;
    double bq[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = tm.row(q);
        bq[q] = row < n ? io.b[row] : 0.0;
        eb = max(eb, (__double2hiint(bq[q]) >> 20) & 0x7ff);
    }
    eb = g.max_int(eb) - 1022 - 57;
    // (b below 2^61 and A x below 2^62, in the finest unit that allows)
    int eo = max(eb - 4, ex4 + sigma - 3);
    long long w[R];
#pragma unroll
    for (int q = 0; q < R; ++q)
        w[q] = to_int(bq[q], -eo) - shr(t[q].hh + t[q].hh + (t[q].m >> 28), eo - ex4 - sigma + 3);
    const Sc res = norm2_full(w, eo, g);
    if (take) {
#pragma unroll
        for (int q = 0; q < R; ++q) Rv[q] = w[q];
        eR = eo;
        bR = 57;
    }
    return res;
}

// The set-up of a solve with Jacobi folded in: whether the system fits (`run`;
// false is returned, and nothing has been overwritten, where no group's does),
// the staged matrix as digits of A D^-1, x~ = D x0, r = b - A x~ and ||b||^2.
//
// A system fits where 57 bits below one scale per vector do for FP64's 53 below
// each entry's own:
//   * the scale of each row's equation, y_i + sum_j |a_ij / a_jj| y_j with y =
//     |b| + |D x0| (to a factor of 2), is at least 2^-12 of the largest y, so that
//     the smallest equation still holds 45 bits of itself; else rows in other units,
//     entries that matter at 1e-6 and 1e-20 alike and parts of a system that hardly
//     meet would lose theirs (A = diag(1, 2^-70), b = (1, 2^-70): x = (1, 0)).
//     folded_finish looks at the solution in the same way. (Right-hand sides drawn
//     from [-1, 1]: none of 2,000,000 3-point systems misses the line; at 2^-8 one in
//     19,000 would, by a corner row, and its whole batch waits for the FP64 code);
//   * BiCGSTAB and CG: each row's diagonal entry exceeds its others by 2^-7 and by
//     2^-9. Below that the Krylov vectors fall and rise by more than the spare bits
//     in a step, and systems that take more iterations than they have rows took up
//     to 4 % more of them (3-point, n = 64; BiCGSTAB with excess 0.001: 93.7 for 89.8
//     in FP64, 0.008: 71.3 for 70.9, 0.016 and more the same; CG 0.0001: 74.8 for
//     74.0, 0.001: 67.9 for 67.7, 0.004 and more the same). GMRES has no line: it
//     starts afresh from the true residual every few steps;
//   * CG: the diagonal is positive and within 2^24 of itself (bbs_fixed_cg.cuh).
enum Method { kBicgstab, kCg, kGmres };
template <int FMT, int SF, Method METHOD, int R, class G>
__device__ __forceinline__ bool folded_setup(const Mat<double>& A, const Mat<double>& S, const SysIO& io, bool valid,
                                             const TeamSmem& sm, G& g, const Team& tm, long long (&X)[R], int& eX,
                                             int& bX, long long (&Rv)[R], int& eR, int& bR, int& sigma, bool& run,
                                             Sc& nb2) {
    const int n = io.n;
    int2* as = in_shared<int2>(S.vals);
    int2* pa = in_shared<int2>(sm.xa);
    int2* pb = in_shared<int2>(sm.xb);
    const bool last = tm.row(R - 1) < n;
    eX = kNone;
    bX = 0;
    // (loops over the caller's rows stay rolled here: this runs once)
    long long* dm = in_shared<long long>(sm.xb);  // 1 / a_ii: its digits,
    int2* de = pa;                                // its exponent beside y_i's biased one, and its FP32 value
    int bad = 0, eb = 0, exm = 0, yleast = 0x7ff, dmost = -100000, dleast = 100000;
#pragma unroll 1
    for (int row = tm.tid; row < n; row += tm.nt) {
        double d = 0.0;
        each_entry<SF>(S, row, [&](int e, int col) {
            if (col == row) d = S.vals[e];
        });
        bad |= normal64(d) ? 0 : 1;
        const Sc di = rcp(unpack(d));
        dm[row] = di.m;
        if (METHOD == kCg) {
            bad |= d > 0.0 ? 0 : 1;
            dmost = max(dmost, di.e);
            dleast = min(dleast, di.e);
        }
        const double xt = d * io.x[row];
        const int yb = (__double2hiint(io.b[row]) >> 20) & 0x7ff;
        const int yx = zero64(xt) ? 0 : max(1, (__double2hiint(xt) >> 20) & 0x7ff);
        de[row] = make_int2((int)((unsigned)di.e << 11) | max(yb, yx), __float_as_int(fabsf(__frcp_rn((float)d))));
        yleast = min(yleast, max(yb, yx));
        eb = max(eb, yb);
        exm = max(exm, yx);
    }
    g.sync();
    int top = 0;  // largest row sum (as the bits of a non-negative FP32, NaN on top)
#pragma unroll 1
    for (int row = tm.tid; row < n; row += tm.nt) {
        float t = 0.0f, u = 0.0f;
        each_entry<SF>(S, row, [&](int e, int col) {
            if (col >= 0) {
                const float v = fabsf((float)S.vals[e]);
                t = fmaf(v, __int_as_float(de[col].y), t);
                if (METHOD != kGmres) u += v;
            }
        });
        top = max(top, __float_as_int(t * 1.0001f) & 0x7fffffff);
        if (METHOD != kGmres)
            bad |= u * __int_as_float(de[row].y) <= 2.0f - (METHOD == kCg ? kExcessCg : kExcess) ? 0 : 1;
    }
    top = g.max_int(bad ? 0x7fffffff : top);
    eb = g.max_int(eb);
    exm = g.max_int(exm);
    yleast = -g.max_int(-yleast);
    const int ym = max(eb, exm);
    const bool xz = exm == 0;  // the guess is zero
    const int spread = METHOD == kCg ? g.max_int(dmost) + g.max_int(-dleast) : 0;
    run = valid && top < __float_as_int(kRowSumMax) && spread <= kDiagonalBits && eb > 623 && eb < 1423 &&
          (xz || (exm > 623 && exm < 1423));
    if (g.any(run && ym - yleast >= kRowScaleBits)) {  // y_i alone does not show it: rare
        int low = 0x7f800000;  // smallest row scale, against 2^ym
#pragma unroll 1
        for (int row = tm.tid; row < n; row += tm.nt) {
            float u = 0.0f;
            each_entry<SF>(S, row, [&](int e, int col) {
                if (col >= 0)
                    u = fmaf(fabsf((float)S.vals[e]) * __int_as_float(de[col].y),
                             __int_as_float(max(127 + (de[col].x & 0x7ff) - ym, 0) << 23), u);
            });
            low = min(low, __float_as_int(u) & 0x7fffffff);
        }
        low = -g.max_int(-low);
        if (ym - yleast >= kRowScaleBits) run = run && low >= __float_as_int(kRowScale);
    }
    if (!g.any(run)) return false;
    sigma = max(1, (top >> 23) - 126);  // row sums < 2^sigma
    const int ebq = eb - 1022 - 57;
    // --- the matrix as digits: A D^-1 2^(60 - sigma), unit diagonal, the
    // quotients to the last bit or two
    const auto digits = [&](double v, int row, int col) {
        long long a = 0;
        if (col == row) {
            a = 1ll << (60 - sigma);
        } else if (col >= 0) {
            const Sc u = unpack(v);
            a = round_shr(mul62(u.m, dm[col]), sigma - 122 - u.e - (de[col].x >> 11));
        }
        return pack(split(a));
    };
#pragma unroll 1
    for (int row = run ? tm.tid : n; row < n; row += tm.nt) {
        if (SF == FMT_DENSE && by_columns(n)) {  // (read again from global memory: not in place)
#pragma unroll 2
            for (int j = 0; j < n; ++j) as[j * n + row] = digits(ldg(A.vals + (size_t)row * n + j), row, j);
        } else {
            each_entry<SF>(S, row, [&](int e, int col) { as[e] = digits(S.vals[e], row, col); });
        }
    }
    g.sync();
    // --- r = b - A x~
    eR = ebq;
    Dot d;
    d.clear();
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = tm.row(q);
        Rv[q] = row < n ? to_int(io.b[row], -ebq) : 0;
        X[q] = 0;
        d.square(split(Rv[q]));
    }
    const Part pt[1] = {part(d)};
    const int pe[1] = {2 * ebq};
    Sc r[1];
    unsigned none = 0;
    g.sums(pt, pe, r, none);
    nb2 = r[0];
    if (g.any(run && !xz)) {
        if (!xz) {
            eX = exm - 1022 - 57;
            bX = 57;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) X[q] = to_int(diag_entry<FMT>(A, tm.row(q)) * io.x[tm.row(q)], -eX);
        }
        true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, !xz, g, tm);
    }
    return true;
}

// The end of such a solve, for the groups with `take` set: x = D^-1 x~ rounded
// to FP64, its residual, and the log. `known`: res2 is the true residual of x~.
// Returns whether the result stands: a system that has converged has to have done
// so as it is returned, and the scales of its rows (setup's, with x~ for y) have
// to be in reach of each other. If not, nothing has been written and FP64 solves
// the system.
template <int FMT, int SF, int R, class G>
__device__ __forceinline__ bool folded_finish(const Mat<double>& A, const Mat<double>& S, const int2* as, int2* pb,
                                              const SysIO& io, int sigma, long long (&X)[R], int& eX, int& bX,
                                              long long (&Rv)[R], int& eR, int& bR, bool take, int iters, int status,
                                              bool known, Sc res2, Sc tau2, Sc nb2, const TeamSmem& sm, G& g,
                                              const Team& tm) {
    if (!g.any(take)) return false;
    const int n = io.n;
    const bool last = tm.row(R - 1) < n;
    long long* xw = in_shared<long long>(sm.xa);  // x~, then the bits of x
    long long* xr = in_shared<long long>(sm.xb);  // x~ of the rounded x
    const bool moved = take && iters > 0;
    // the scales of the rows: |x~_i| + |b_i| shows nearly always that they are
    int hi = -100000, lo = 100000;
#pragma unroll
    for (int q = 0; q < R; ++q)
        if (q + 1 < R || last) {
            xw[tm.row(q)] = X[q];
            const int b = ((__double2hiint(io.b[tm.row(q)]) >> 20) & 0x7ff) - 1022;
            const int l = max(64 - __clzll(X[q] ^ (X[q] >> 63)) + eX, b);
            hi = max(hi, l);
            lo = min(lo, l);
        }
    hi = g.max_int(hi);
    lo = -g.max_int(-lo);
#pragma unroll 1
    for (int row = moved ? tm.tid : n; row < n; row += tm.nt) {
        const Sc d = unpack(diag_entry<FMT>(A, row));
        const double x = to_double(mul(normal(xw[row], eX), rcp(d)));
        xw[row] = __double_as_longlong(x);
        const Sc u = unpack(x);
        xr[row] = round_shr(mul62(u.m, d.m), eX - u.e - d.e - 62);
    }
    // Rounding moves the residual by at most 2^-53 of the row sums of |A~| |x~|:
    // below 2^(sigma + hi - 53 + 6) in the norm (2,048 rows). Where that is below 2^-12 of
    // the known residual, the log states it, and a converged system has converged
    // unless the two are as close to the tolerance.
    const int slack = 2 * (sigma + hi - 53 + 6 + 12);
    const bool exact = !known || (moved && (res2.e + 61 < slack || (status == ST_CONVERGED && !le(res2, normal(tau2.m - (tau2.m >> 11), tau2.e)))));
    const bool wide = hi - lo > kRowScaleBits;
    if (g.any(take && (exact || wide))) {
        if (moved) {
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) X[q] = xr[tm.row(q)];
        }
        int ey = 0;
        const Sc res = true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, false, g, tm, &ey);
        if (exact) res2 = res;
        if (g.any(take && wide)) {
            Abs t[R];
            spmv_sums<SF, 64>(S, as, pb, t, 0, tm);
            int h = -100000, l = 100000;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    const int b = ((__double2hiint(io.b[tm.row(q)]) >> 20) & 0x7ff) - 1022;
                    const int v = max(64 - __clzll(t[q].hh) + ey + sigma - 2, b);
                    h = max(h, v);
                    l = min(l, v);
                }
            h = g.max_int(h);
            l = -g.max_int(-l);
            if (wide) {
                hi = h;
                lo = l;
            }
        }
    }
    const bool good = take && hi - lo <= kRowScaleBits + 1 && finite(res2) &&
                      (status != ST_CONVERGED || le(res2, tau2));
    if (good) {
#pragma unroll 1
        for (int row = moved ? tm.tid : n; row < n; row += tm.nt) io.x[row] = __longlong_as_double(xw[row]);
        if (tm.tid == 0) {
            *io.iters = iters;
            *io.rel_res = sqrt(to_double(res2) / to_double(nb2));
            *io.status = status;
            if (io.inner != nullptr) *io.inner = 0;
        }
    }
    return good;
}

// --------------------------------------------------------------- BiCGSTAB

// BiCGSTAB with Jacobi folded into the staged matrix, as
// bicgstab_scaled_system: the method, its tests and its scalars are the same;
// the vectors are block fixed point. A: the system in its own format FMT
// (diagonal lookups), S: the staged copy in format SF, whose values this
// overwrites with digits once the system has qualified. `valid` is false for
// a group without a system of its own (it reads, and never writes). A system
// that FP64 has to solve (one that does not fit, or has broken down, stagnated or
// met a non-finite scalar here) has its x and its log untouched.
template <int FMT, int SF, int R, class G>
__device__ __forceinline__ Fit bicgstab_fixed(const Mat<double>& A, const Mat<double>& S, const SysIO& io, bool valid,
                                               const SolveCfg& C, const TeamSmem& sm, G g, const Team& team) {
    const int n = io.n;
    Team tm = team;
    if (G::kLanes != 0) tm.nt = G::kLanes;  // (known to the compiler)
    int2* as = in_shared<int2>(S.vals);
    int2* pa = in_shared<int2>(sm.xa);  // p
    int2* pb = in_shared<int2>(sm.xb);  // s, and x~ for true residuals

    long long X[R], Rv[R];  // x~ = D x, r (then s)
    Dig rh[R], v[R];
    int eX = kNone, bX = 0, eR, bR, sigma;
    bool run;
    Sc nb2;
    if (!folded_setup<FMT, SF, kBicgstab>(A, S, io, valid, sm, g, tm, X, eX, bX, Rv, eR, bR, sigma, run, nb2)) {
        // (the block's other warps count on this one at their barriers)
        for (int it = 1; it <= C.max_iters && g.live(false); ++it) {
        }
        return kUnfit;
    }
    const bool last = tm.row(R - 1) < n;  // only a lane's last row may lie past the end
    const Sc tol2 = unpack(C.tol * C.tol), tau2 = C.tol_type == 1 ? mul(tol2, nb2) : tol2;
    Sc rr = norm2_full(Rv, eR, g);
    bR = 57;
#pragma unroll
    for (int q = 0; q < R; ++q) rh[q] = split(Rv[q]);
    int eH = eR;  // r^ = r
    int status = -1, iters = 0, restarts = 0;
    Sc res2 = rr;
    bool active = run;
    if (active && le(rr, tau2)) {
        status = ST_CONVERGED;
        active = false;
    }
    Sc rho = rr, alpha = one(), omega = one(), cfac = one();
    int eP = kNone, bP = 0, eV = kNone, bV = 0;
    g.sync();  // every lane is done reading pa
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = tm.row(q);
        v[q] = Dig{0, 0};
        if (row < n) pa[row] = make_int2(0, 0);  // p = 0
    }

    const auto residual = [&](bool take) -> Sc {
        return true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, take, g, tm);
    };

    for (int it = 1; it <= C.max_iters; ++it) {
        if (!g.live(active)) break;
        if (!g.any(active)) continue;
        if (active) {
            iters = it;
            if (!finite(rho)) {
                status = ST_NAN;
                active = false;
            } else if (zero(rho)) {
                status = ST_BREAKDOWN;
                active = false;
            }
        }
        unsigned op;
        {  // r to 56 bits, p = r + beta (p - omega v)
            fill_up(Rv, eR, bR, g);
            const Sc beta = mul(rho, cfac), bo = neg(mul(beta, omega));
            const int eo = max(max(eR + max(0, bR - 55), eP + ex(beta) + max(-2, bP - 55)),
                               eV + ex(bo) + max(-2, bV - 55));
            const Dig c1 = coef(beta, eP, eo), c2 = coef(bo, eV, eo);
            long long t[R];
#pragma unroll
            for (int q = 0; q < R; ++q) t[q] = Rv[q];
            shr_rows(t, eo - eR, g);
            op = 0;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    Sum s{t[q], 1 << 28};
                    s.add(c1, dig(pa[tm.row(q)]));
                    s.add(c2, v[q]);
                    const Dig f = split(s.value());
                    pa[tm.row(q)] = pack(f);
                    op |= mag(f.hi);
                }
            eP = eo;
        }
        g.sync();
        spmv_fixed<SF, R>(S, as, pa, v, tm);
        eV = eP + sigma - 2;
        Sc sigm;
        {
            Dot d{0, 0, 0};
            unsigned ov = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                d.add(rh[q], v[q]);
                ov |= mag(v[q].hi);
            }
            const Part pt[1] = {part(d)};
            const int pe[1] = {eH + eV};
            Sc r[1];
            unsigned o = masks(op, ov);
            g.sums(pt, pe, r, o);
            sigm = r[0];
            bP = bits_first(o);
            bV = bits_second(o);
        }
        if (active) {
            if (!finite(sigm)) {
                status = ST_NAN;
                active = false;
            } else if (zero(sigm)) {
                status = ST_BREAKDOWN;
                active = false;
            }
        }
        alpha = mul(rho, rcp(sigm));
        int eS;
        {  // s = r - alpha v
            eS = max(eR + max(0, bR - 56), eV + ex(alpha) + max(-2, bV - 56));
            const Dig c = coef(neg(alpha), eV, eS);
            shr_rows(Rv, eS - eR, g);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                Sum s{Rv[q], 1 << 28};
                s.add(c, v[q]);
                Rv[q] = s.value();
                if (q + 1 < R || last) pb[tm.row(q)] = pack(split(Rv[q]));
            }
        }
        g.sync();
        Dig t[R];
        spmv_fixed<SF, R>(S, as, pb, t, tm);
        const int eT = eS + sigma - 2;
        Sc ss, tt, ts;
        int bS, bT;
        {
            Dot ds{0, 0, 0}, dx{0, 0, 0};
            long long carry;
            const Dot dt = dot_wide(t, carry);
            unsigned os = 0, ot = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const Dig f = split(Rv[q]);
                ds.square(f);
                dx.add(t[q], f);
                os |= mag(f.hi);
                ot |= mag(t[q].hi);
            }
            const Part pt[3] = {part(ds), part(dt, carry), part(dx)};
            const int pe[3] = {2 * eS, 2 * eT, eS + eT};
            Sc r[3];
            unsigned o = masks(os, ot);
            g.sums(pt, pe, r, o);
            ss = r[0];
            tt = r[1];
            ts = r[2];
            bS = bits_first(o);
            bT = bits_second(o);
        }
        if (active && !finite(ss)) {
            status = ST_NAN;
            active = false;
        }
        const bool half = active && le(ss, tau2);
        bool full = active && !half;
        bool cand = half;
        Sc rho_next{0, kNone};
        if (full && (!finite(tt) || !finite(ts))) {
            status = ST_NAN;
            active = false;
            full = false;
        }
        // omega = ts / tt (0 for tt = 0) and the next beta's alpha / (rho omega) =
        // (alpha tt) / (rho ts)
        Sc om = zero(tt) ? Sc{0, kNone} : mul(ts, rcp(tt));
        if (full) {
            omega = om;
            cfac = mul(mul(alpha, tt), rcp(mul(rho, ts)));
        }
        {  // x~ += alpha p + omega s (a half step: alpha p), kept to 61 bits
            const Sc oms = full ? om : Sc{0, kNone};
            const int eo = max(max(eX + max(0, bX - 59), eP + ex(alpha) - 2), eS + ex(oms) - 2);
            const bool move = half || full;  // (a system that has stopped keeps its x~: both multipliers are 0)
            Dig c1 = coef(alpha, eP, eo), c2 = coef(oms, eS, eo);
            if (!move) c1 = c2 = Dig{0, 0};
            if (!full) c2 = Dig{0, 0};
            shr_rows(X, move ? eo - eX : 0, g);
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    Sum s{X[q], 1 << 28};
                    s.add(c1, dig(pa[tm.row(q)]));
                    s.add(c2, split(Rv[q]));
                    X[q] = s.value();
                }
            if (move) eX = eo;
        }
        {  // r = s - omega t
            eR = max(eS + max(0, bS - 56), eT + ex(om) + max(-2, bT - 56));
            const Dig c = coef(neg(om), eT, eR);
            Dot dr{0, 0, 0}, dh{0, 0, 0};
            unsigned orr = 0, ox = 0;
            shr_rows(Rv, eR - eS, g);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                Sum s{Rv[q], 1 << 28};
                s.add(c, t[q]);
                Rv[q] = s.value();
                const Dig f = split(Rv[q]);
                dr.square(f);
                dh.add(rh[q], f);
                orr |= mag(f.hi);
                ox |= mag((int)(X[q] >> 32));
            }
            const Part pt[2] = {part(dr), part(dh)};
            const int pe[2] = {2 * eR, eH + eR};
            Sc r[2];
            unsigned o = masks(orr, ox);
            g.sums(pt, pe, r, o);
            rr = r[0];
            rho_next = r[1];
            bR = bits_first(o);
            bX = bits_second(o) + 3;  // (of the upper words)
        }
        if (full) {
            if (!finite(rr)) {
                status = ST_NAN;
                active = false;
            } else {
                cand = le(rr, tau2);
            }
        }
        bool restarted = false;
        if (g.any(cand)) {
            const Sc res = residual(cand);
            if (cand) {
                res2 = res;
                if (!finite(res)) {
                    status = ST_NAN;
                    active = false;
                } else if (le(res, tau2)) {
                    status = ST_CONVERGED;
                    active = false;
                } else if (++restarts > kMaxRestarts) {
                    status = kStagnated;
                    active = false;
                } else {
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        const int row = tm.row(q);
                        rh[q] = split(Rv[q]);
                        v[q] = Dig{0, 0};
                        if (row < n) pa[row] = make_int2(0, 0);
                    }
                    eH = eR;
                    eP = eV = kNone;
                    bP = bV = 0;
                    rho = res;
                    alpha = omega = cfac = one();
                    restarted = true;
                }
            }
        }
        if (active && !restarted) {
            if (zero(omega)) {
                status = ST_BREAKDOWN;
                active = false;
            } else {
                rho = rho_next;
            }
        }
    }
    if (active) status = ST_MAX_ITER;
    return folded_finish<FMT, SF>(A, S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, run && accepted(status), iters, status,
                                  status == ST_CONVERGED, res2, tau2, nb2, sm, g, tm)
               ? kDone
               : run ? kLeft : kUnfit;
}

}  // namespace fx

// --------------------------------------------------- teams of whole warps

// BiCGSTAB with Jacobi on staged values (`count` of them): block fixed point, or
// FP64 for the systems that do not fit it (and for teams of more warps than the
// fixed-point reductions hold).
template <int FMT, int R>
__device__ __forceinline__ void bicgstab_staged_jacobi(const Op<FMT, R, double, double>& op, size_t count,
                                                       const SysIO& io, const SolveCfg& C, const TeamSmem& sm,
                                                       const Team& tm) {
    if (tm.nwarps <= fx::kMaxWarps) {
        const Mat<double> S{op.as, op.A.row_ptrs, op.A.cols, op.A.n, op.A.k};
        const fx::Warps g{tm, reinterpret_cast<unsigned char*>(sm.red), 0};
        const fx::Fit fit = fx::bicgstab_fixed<FMT, FMT, R>(op.A, S, io, true, C, sm, g, tm);
        if (fit == fx::kDone) return;
        tm.sync();
        if (fit == fx::kLeft) make_op<FMT, R>(op.A, count, const_cast<double*>(op.as), tm);
    }
    bicgstab_scaled_system<FMT, R>(op, io, C, sm, tm);
}

// No cap on the registers beyond the block's own: at 128, which kept more FP64
// warps resident at 5-6 rows per thread, the fixed-point code spills (BiCGSTAB,
// n = 324, 9-point, 2 warps: 4,000 systems 2.02 -> 1.59 ms, 117 systems 376 ->
// 217 us; the FP64 kernel took 2.51 ms and 368 us).
template <int FMT, int R>
__global__ void __launch_bounds__(max_threads_for(R), 1)
    bicgstab_folded_kernel(const SolveParams P) {
    extern __shared__ __align__(16) unsigned char raw[];
    const Team tm = Team::block();
    const int sys = blockIdx.x;
    const auto op = make_op<FMT, R>(P, sys, raw, tm);
    bicgstab_staged_jacobi<FMT, R>(op, P.vps, sys_io(P, sys), solve_cfg(P, sys), team_smem(raw, P.n_pad), tm);
}
}  // namespace bbs
