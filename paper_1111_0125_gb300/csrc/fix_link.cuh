// FP64 links as the integer Dslash reads them (fix64.cuh), without loss.
//
// A real number u of a link, |u| < 2, takes the 8 bytes of its double as two
// words: u rounded to a multiple of 2^-57 is h 2^-29 + l 2^-57, -2^27 <= l < 2^27; h lies
// in the upper 31 bits of the first word and l in the upper 28 of the second.
// The five bits left over of each number of a link together hold what the
// rounding took off: a number whose size cut to 2^-57 has b significant bits
// lacks the last 53 - b of its significand (numbers of 1/32 or more lack none),
// and one bit more where the rounded value is a power of two (whether it was
// carried there); one that is cut to zero is zero in h and l and takes two
// bits if it is zero and 65 otherwise.  Random SU(3) links need 2 to 4 bits on
// average; the 82 (18-real) or 52 (12-real) that are there suffice for all but
// one in about 1e10 links exp(i eps H) with eps >= 0.2.  A field with a link that
// needs more (nearly all links close to 1, say) keeps its doubles.
//
// The low four bits of the second word of numbers 0 and 1 hold the link's
// spreads, in eighths: with the six numbers of a row in order of size, the sum
// of all but the largest, the least of the three rows; and the same for the
// columns.
#pragma once

#include <cuda_runtime.h>
#include <string.h>

namespace stg {

// left-over bits of a link of N numbers, and reading and writing them
template <int N> struct FixPool {
    static constexpr int size = 2 + 5 * (N - 2);
    unsigned long long lo = 0, hi = 0;
    int at = 0;
    __host__ __device__ void put(unsigned long long v, int n)
    {
        if (n > 0 && at + n <= size) {
            if (at < 64) {
                lo |= v << at;
                if (at + n > 64) hi |= v >> (64 - at);
            } else {
                hi |= v << (at - 64);
            }
        }
        at += n;
    }
    __host__ __device__ unsigned long long get(int n)
    {
        if (n <= 0) return 0;
        unsigned long long v = at < 64 ? lo >> at : hi >> (at - 64);
        if (at > 0 && at < 64 && at + n > 64) v |= hi << (64 - at);
        at += n;
        return n < 64 ? v & ((1ull << n) - 1) : v;
    }
    // the bits of number r: those of the second word and, above, that of the first
    __host__ __device__ unsigned of(int r) const
    {
        if (r < 2) return (unsigned)(lo >> r & 1) << 4;
        const int b = 2 + 5 * (r - 2);
        unsigned long long v = b < 64 ? lo >> b : hi >> (b - 64);
        if (b < 64 && b + 5 > 64) v |= hi << (64 - b);
        return (unsigned)v & 31u;
    }
    __host__ __device__ void set(int r, unsigned v)
    {
        if (r < 2) {
            lo |= (unsigned long long)(v >> 4 & 1) << r;
            return;
        }
        const int b = 2 + 5 * (r - 2);
        if (b < 64) {
            lo |= (unsigned long long)v << b;
            if (b + 5 > 64) hi |= (unsigned long long)v >> (64 - b);
        } else {
            hi |= (unsigned long long)v << (b - 64);
        }
    }
};

__host__ __device__ inline unsigned long long fix_bits(double u)
{
    unsigned long long b;
    memcpy(&b, &u, sizeof(b));
    return b;
}

__host__ __device__ inline int fix_width(unsigned long long x)  // significant bits of x > 0
{
#ifdef __CUDA_ARCH__
    return 64 - __clzll((long long)x);
#else
    return 64 - __builtin_clzll(x);
#endif
}

// |u| cut to 2^-57, in those units
__host__ __device__ inline unsigned long long fix_units(unsigned long long bits)
{
    const int e = (int)(bits >> 52 & 0x7ff) - 1018;
    const unsigned long long m = (bits & 0xfffffffffffffull) | 1ull << 52;
    return e >= 0 ? m << e : e > -53 ? m >> -e : 0ull;
}

// the same rounded to the nearest (half away from zero; not up from zero);
// lack: the bits of the significand below
__host__ __device__ inline unsigned long long fix_round(unsigned long long bits, int &lack)
{
    const unsigned long long x = fix_units(bits);
    lack = x ? 53 - fix_width(x) : 0;
    return lack > 0 ? x + (bits >> (lack - 1) & 1) : x;
}

// Numbers u (each below 2 in size) to words; false, and nothing written, where
// they do not fit.  row, col: the spreads, 0 to 15.
template <int N> __host__ __device__ inline bool fix_encode(const double *u, unsigned row, unsigned col, int2 *w)
{
    FixPool<N> pool;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const unsigned long long b = fix_bits(u[r]), x = fix_units(b);
        if (x == 0) {
            if (b << 1 == 0) {
                pool.put(b >> 63 << 1, 2);
            } else {
                pool.put(1, 1);
                pool.put(b, 64);
            }
        } else {
            int lack;
            const unsigned long long y = fix_round(b, lack);
            if ((y & (y - 1)) == 0 && fix_width(y) <= 53) pool.put(fix_width(y) != fix_width(x), 1);
            if (lack > 0) pool.put(b & ((1ull << lack) - 1), lack);
        }
    }
    if (pool.at > FixPool<N>::size) return false;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const unsigned long long b = fix_bits(u[r]);
        int lack;
        const long long y = (long long)fix_round(b, lack), x = b >> 63 ? -y : y;
        const int h = (int)((x + (1 << 27)) >> 28), l = (int)(x - ((long long)h << 28));
        const unsigned p = pool.of(r);
        w[r].x = (int)((unsigned)h << 1 | p >> 4);
        w[r].y = (int)((unsigned)l << 4 | (r == 0 ? row : r == 1 ? col : p & 15u));
    }
    return true;
}

// the numbers, bit for bit
template <int N> __host__ __device__ inline void fix_decode(const int2 *w, double *u)
{
    FixPool<N> pool;
#pragma unroll
    for (int r = 0; r < N; ++r) pool.set(r, (unsigned)(w[r].y & 15) | (unsigned)(w[r].x & 1) << 4);
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const long long v = ((long long)(w[r].x >> 1) << 28) + (w[r].y >> 4);
        unsigned long long b;
        if (v == 0) {
            b = pool.get(1) ? pool.get(64) : pool.get(1) << 63;
        } else {
            const unsigned long long y = v < 0 ? (unsigned long long)-v : (unsigned long long)v;
            int n = fix_width(y);
            if ((y & (y - 1)) == 0 && n <= 53) n -= (int)pool.get(1);
            const int lack = 53 - n;
            unsigned long long m = y >> (lack < 0 ? -lack : 0);
            if (lack > 0) {
                const unsigned long long rest = pool.get(lack);
                m = (y - (rest >> (lack - 1))) << lack | rest;
            }
            b = (v < 0 ? 1ull << 63 : 0ull) | (unsigned long long)(n + 965) << 52 | (m & 0xfffffffffffffull);
        }
        memcpy(&u[r], &b, sizeof(b));
    }
}

// The spreads of a matrix given by the sizes of its numbers, a[row][column][re, im],
// rounded down.
__host__ __device__ inline void fix_spreads(const float (&a)[3][3][2], unsigned &row, unsigned &col)
{
    float s[2] = {2.f, 2.f};
    for (int k = 0; k < 3; ++k)
        for (int way = 0; way < 2; ++way) {
            float sum = 0.f, top = 0.f;
            for (int j = 0; j < 3; ++j)
                for (int z = 0; z < 2; ++z) {
                    const float v = way ? a[j][k][z] : a[k][j][z];
                    sum += v;
                    top = v > top ? v : top;
                }
            s[way] = sum - top < s[way] ? sum - top : s[way];
        }
    const float up = 8.f, slack = 1e-3f;
    row = s[0] > slack ? (unsigned)((s[0] - slack) * up) : 0u;
    col = s[1] > slack ? (unsigned)((s[1] - slack) * up) : 0u;
    row = row > 15u ? 15u : row;
    col = col > 15u ? 15u : col;
}

}  // namespace stg
