// Host check of the one-range activity test (csrc/asse_cyclic.h) against
// Algorithm 1 and Algorithm 2 written out per value: every k in 1..127, k',
// ACT and stored value, then whole words of fields with tests of their own, at
// every field width.  Prints the number of mismatches and "ok" when there are
// none.
#include <cstdint>
#include <cstdio>

#include <cuda_runtime.h>

#include "asse_cyclic.h"

using namespace asse;

static uint32_t state = 2463534242u;
static uint32_t rnd(uint32_t n)
{
    state ^= state << 13;
    state ^= state >> 17;
    state ^= state << 5;
    return (uint32_t)(((uint64_t)state * n) >> 32);
}

static uint32_t width(bool ace, uint32_t k)
{
    const uint32_t v = ace ? k + 1 : 2 * k + 1;
    uint32_t b = 0;
    while ((1u << b) < v)
        b++;
    return b == 0 ? 1 : b;
}

static bool active(bool ace, uint32_t k, uint32_t kp, uint32_t act, uint32_t v)
{
    if (ace)
        return v >= k - kp + 1;
    if (v >= 2 * k)
        return false;
    for (uint32_t a = 0; a < kp; a++)
        if ((act + 2 * k - a) % (2 * k) == v)
            return true;
    return false;
}

static bool cleared(uint32_t k, uint32_t act, uint32_t v)
{
    if (act == 0)
        return v <= k;
    if (act == k)
        return v == 0 || (v >= k && v < 2 * k);
    return false;
}

static bool pass(CyclicRange r, uint32_t vmax, uint32_t v, uint32_t w)
{
    return ((v + r.c) & ((1u << w) - 1)) <= r.h && v <= vmax;
}

template <int WB, bool BG>
static long words(bool ace, uint32_t k)
{
    using L = CyclicLayout<WB, BG>;
    constexpr uint32_t F = L::F;
    long bad = 0;
    const uint32_t top = ace ? k : 2 * k, vmax = cyclic_vmax(ace, k, L::W);
    for (int it = 0; it < 400; it++) {
        typename L::Entry d = L::empty();
        uint32_t w = 0, want = 0, full = 0;
        for (uint32_t j = 0; j < F; j++) {
            uint32_t v = rnd(top + 1);
            const uint32_t act = rnd(2 * k), kp = 1 + rnd(k), kind = rnd(8);
            bool on;
            if (kind == 0) {  // past g
                v = 0;
                L::put(d, j, cyclic_none_past_g());
                on = false;
            } else if (kind < 3 && !ace) {
                const uint32_t a = kind == 1 ? (rnd(2) ? k : 0) : act;
                L::put(d, j, cyclic_cleared(k, a, L::W));
                on = cleared(k, a, v);
            } else {
                L::put(d, j, cyclic_active(ace, k, kp, act, L::W));
                on = active(ace, k, kp, act, v);
            }
            w |= v << (j * WB);
            want |= (uint32_t)on << j;
            full |= on ? ((1u << WB) - 1) << (j * WB) : 0u;
        }
        const uint32_t r = L::test(w, d, L::limit(vmax));
        bad += L::compress(r) != want;
        bad += L::widen(r) != full;
        bad += __builtin_popcount(r) != __builtin_popcount(want);
    }
    return bad;
}

int main()
{
    long bad = 0, checked = 0;
    for (uint32_t ace = 0; ace < 2; ace++)
        for (uint32_t k = 1; k <= 127; k++) {
            const uint32_t w = width(ace, k), vmax = cyclic_vmax(ace, k, w), top = ace ? k : 2 * k;
            for (uint32_t act = 0; act < (ace ? 1 : 2 * k); act++) {
                for (uint32_t kp = 1; kp <= k; kp++) {
                    const CyclicRange r = cyclic_active(ace, k, kp, act, w);
                    if (r.h >= (1u << w) || r.c >= (1u << w))
                        bad++;
                    // the members of the window are act, act-1, ..: mark them once
                    bool in[256] = {};
                    for (uint32_t a = 0; a < kp; a++)
                        in[ace ? k - a : (act + 2 * k - a) % (2 * k)] = true;
                    for (uint32_t v = 0; v <= top; v++, checked++)
                        bad += pass(r, vmax, v, w) != in[v];
                }
                if (!ace)
                    for (uint32_t v = 0; v <= top; v++, checked++)
                        bad += pass(cyclic_cleared(k, act, w), vmax, v, w) != cleared(k, act, v);
            }
            switch (w) {
            case 1: bad += words<1, false>(ace, k); break;
            case 2: bad += words<2, false>(ace, k); break;
            case 3: bad += words<3, false>(ace, k); break;
            case 4: bad += words<4, false>(ace, k); break;
            case 5: bad += words<5, false>(ace, k); break;
            case 6: bad += words<6, false>(ace, k); break;
            case 7: bad += words<8, true>(ace, k); break;
            case 8: bad += words<8, false>(ace, k); break;
            }
        }
    printf("checked %ld, bad %ld\n%s\n", checked, bad, bad ? "mismatch" : "ok");
    return bad != 0;
}
