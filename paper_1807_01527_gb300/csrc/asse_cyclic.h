// The activity test of the scan and of asse_estimate as one cyclic range.
//
// The active values of a field are the window act-k'+1 .. act taken mod 2k,
// out of 0 .. 2k-1; 2k means inactive.  With l the window's low end (mod 2k),
// t = (v - l) mod 2^w maps it to 0 .. h: h = k'-1 where it does not wrap past
// 2k-1, and 2^w - 2k + k' - 1 where it does, the gap that the unused values
// 2k .. 2^w - 1 leave in the middle then holding only v = 2k.  So a field is
// active iff t <= h and v <= 2k-1: one addition of 2^w - l and two
// comparisons, against two comparisons for each of two plain ranges.  Aging
// counters (active iff v >= k-k'+1) fit the same test with every v allowed,
// Algorithm 2's values to clear are such windows too (0..k, and k..2k-1 with
// 0), and so is a test no field passes.
//
// The even and the odd fields of a word are tested separately, each field
// then having a guard bit above it: a difference keeps the guard iff it is
// not negative, with no borrow between fields.  The odd group stays in place
// where the word has a bit to spare above its last field, else it is shifted
// down by one field.  Byte-wide fields holding seven-bit values have the guard
// bit inside the field and are tested all four at once.  Host and device code
// (the host build checks it against Algorithms 1 and 2 for every k, k', ACT
// and value).
#pragma once

#include <cstdint>

#include <vector_types.h>

#if defined(__CUDACC__)
#define ASSE_CYCLIC_FN __host__ __device__ __forceinline__
#else
#define ASSE_CYCLIC_FN inline
#endif

namespace asse {

// One field's test: v passes iff ((v + c) mod 2^w) <= h (and v <= vmax, the
// same for every field of a pool).
struct CyclicRange {
    uint32_t c, h;
};

// Largest value that may pass: 2k-1, or any for aging counters.
ASSE_CYCLIC_FN uint32_t cyclic_vmax(bool ace, uint32_t k, uint32_t w)
{
    return ace ? (1u << w) - 1 : 2 * k - 1;
}

// The values low .. low+n-1 mod 2k (n in 1 .. 2k), of fields of w bits.
ASSE_CYCLIC_FN CyclicRange cyclic_window(uint32_t k, uint32_t low, uint32_t n, uint32_t w)
{
    const uint32_t m = 1u << w;
    return CyclicRange{(m - low) & (m - 1), low + n <= 2 * k ? n - 1 : m - 2 * k + n - 1};
}

// Algorithm 1: active in the latest kp slices.
ASSE_CYCLIC_FN CyclicRange cyclic_active(bool ace, uint32_t k, uint32_t kp, uint32_t act, uint32_t w)
{
    const uint32_t m = 1u << w;
    if (ace)
        return CyclicRange{(m - (k + 1 - kp)) & (m - 1), kp - 1};
    return cyclic_window(k, act + 1 >= kp ? act + 1 - kp : act + 2 * k + 1 - kp, kp, w);
}

// No value passes (a field past g, whose stored value is 0).
ASSE_CYCLIC_FN CyclicRange cyclic_none_past_g() { return CyclicRange{1, 0}; }

// Algorithm 2: the values a timestamp field of new ACT act loses.
ASSE_CYCLIC_FN CyclicRange cyclic_cleared(uint32_t k, uint32_t act, uint32_t w)
{
    if (act == 0)
        return cyclic_window(k, 0, k + 1, w);
    if (act == k)
        return cyclic_window(k, k, k + 1, w);
    return CyclicRange{(1u << w) - 2 * k, 0};  // v + c = 2^w only for v = 2k, which never passes
}

// Words of WB-bit fields, even and odd group.
template <int WB>
struct Cyclic {
    static constexpr uint32_t F = 32 / WB;
    static constexpr uint32_t FM = (1u << WB) - 1;
    static constexpr bool IN_PLACE = F * WB < 32;  // the last field's guard bit exists
    static constexpr uint32_t SHIFT = IN_PLACE ? 0 : WB;  // the odd group is shifted down by
    static constexpr uint32_t at(uint32_t j) { return j * WB - (j & 1 ? SHIFT : 0); }
    static constexpr uint32_t fields(uint32_t odd)
    {
        uint32_t m = 0;
        for (uint32_t j = odd; j < F; j += 2)
            m |= FM << at(j);
        return m;
    }
    static constexpr uint32_t guards(uint32_t odd)
    {
        uint32_t m = 0;
        for (uint32_t j = odd; j < F; j += 2)
            m |= 1u << (at(j) + WB);
        return m;
    }
    static constexpr uint32_t ME = fields(0), MO = fields(1), HE = guards(0), HO = guards(1);

    // (c, h | guard) of the even fields in x, y and of the odd ones in z, w.
    using Entry = uint4;
    static ASSE_CYCLIC_FN Entry empty() { return Entry{0, 0, 0, 0}; }
    static ASSE_CYCLIC_FN void put(Entry &d, uint32_t j, CyclicRange r)
    {
        const uint32_t p = j * WB - (j & 1 ? SHIFT : 0);
        if (j & 1) {
            d.z |= r.c << p;
            d.w |= (r.h | (1u << WB)) << p;
        } else {
            d.x |= r.c << p;
            d.y |= (r.h | (1u << WB)) << p;
        }
    }
    // vmax with guards, in both groups.
    struct Limit {
        uint32_t e, o;
    };
    static ASSE_CYCLIC_FN Limit limit(uint32_t vmax)
    {
        Limit l{0, 0};
        for (uint32_t j = 0; j < F; j++)
            (j & 1 ? l.o : l.e) |= (vmax | (1u << WB)) << (j * WB - (j & 1 ? SHIFT : 0));
        return l;
    }
    // One bit of the result per field of w that passes, at bit(j).
    static ASSE_CYCLIC_FN uint32_t test(uint32_t w, const Entry &d, const Limit &l)
    {
        const uint32_t xe = w & ME, xo = (w >> SHIFT) & MO;
        const uint32_t te = (xe + d.x) & ME, to = (xo + d.z) & MO;
        const uint32_t e = (d.y - te) & (l.e - xe), o = (d.w - to) & (l.o - xo);
        if constexpr (IN_PLACE)
            return (e & HE) | (o & HO);
        else
            return (e & HE) | ((o & HO) >> 1);
    }
    static constexpr uint32_t bit(uint32_t j) { return at(j) + WB - (j & 1 ? !IN_PLACE : 0); }
    // Field j (bit j) set iff its bit is set in the result r of test().
    static ASSE_CYCLIC_FN uint32_t compress(uint32_t r)
    {
        uint32_t m = 0;
        for (uint32_t j = 0; j < F; j++)
            m |= ((r >> (j * WB - (j & 1 ? SHIFT : 0) + WB - (j & 1 ? !IN_PLACE : 0))) & 1u) << j;
        return m;
    }
    // The fields of the result r as full fields of the word.
    static ASSE_CYCLIC_FN uint32_t widen(uint32_t r)
    {
        if constexpr (IN_PLACE)
            return (r >> WB) * FM;  // guards lie one field above their fields, at least a field apart
        else
            return ((r & HE) >> WB) * FM | ((r & (HO >> 1)) >> (WB - 1)) * FM << WB;
    }
};

// Byte-wide fields of values below 128.
struct CyclicBytes {
    static constexpr uint32_t G = 0x80808080u;
    using Entry = uint2;  // (c, h | 0x80) per byte
    static ASSE_CYCLIC_FN Entry empty() { return Entry{0, 0}; }
    static ASSE_CYCLIC_FN void put(Entry &d, uint32_t j, CyclicRange r)
    {
        d.x |= r.c << (8 * j);
        d.y |= (r.h | 0x80u) << (8 * j);
    }
    using Limit = uint32_t;
    static ASSE_CYCLIC_FN Limit limit(uint32_t vmax) { return (vmax | 0x80u) * 0x01010101u; }
    static ASSE_CYCLIC_FN uint32_t test(uint32_t w, const Entry &d, Limit l)
    {
        return (d.y - ((w + d.x) & ~G)) & (l - w) & G;
    }
    static ASSE_CYCLIC_FN uint32_t compress(uint32_t r)
    {
        return ((r >> 7) | (r >> 14) | (r >> 21) | (r >> 28)) & 0xFu;
    }
    static ASSE_CYCLIC_FN uint32_t widen(uint32_t r) { return (r >> 7) * 0xFFu; }
};

// The field layout of a kernel of WB-bit fields, BG: byte-wide with values
// below 128 (the test's arithmetic is then of seven-bit fields).
template <int WB, bool BG>
struct CyclicLayout : Cyclic<WB> {
    static constexpr uint32_t W = WB;
};
template <>
struct CyclicLayout<8, true> : CyclicBytes {
    static constexpr uint32_t W = 7, F = 4;
};

}  // namespace asse
