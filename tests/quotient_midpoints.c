/* The quotient of binary32 numbers as the draws form it (su2_device.cuh,
 * div_in_range), over every pair whose quotient lies so close to the middle of
 * two binary32 numbers that its refinement could round the wrong way.
 *
 * With y = RN(1/b), q = RN(a y), r = RN(a - b q), z = RN(q + r y), the number
 * that z rounds is within 8 u^2 of a/b for a quotient in [1, 2), u = 2^-24: q is
 * within 4 u + of a/b, and r and y carry a relative error of u each.  The middle
 * M u (M odd, 25 bits) of two numbers is at |d| u / B from a/b, where
 * a 2^s - M B = d in the integer significands a, B of 24 bits, s = 24 (a >= B) or
 * 25 (a < B).  As B < 2^24, only |d| <= 8 can matter; every case with |d| <= 12
 * is formed by solving for M modulo 2^s, and z compared with the quotient. */
#include <math.h>
#include <stdint.h>
#include <stdio.h>

int main(void)
{
    long cases = 0, wrong = 0;
    for (uint32_t B = 1u << 23; B < 1u << 24; ++B) {
        const float b = (float)B, y = 1.0f / b;
        int twos = 0;
        while (!((B >> twos) & 1u)) ++twos;
        const uint32_t odd = B >> twos;
        uint32_t inverse = odd; /* of odd, modulo 2^32 */
        for (int k = 0; k < 5; ++k) inverse *= 2u - odd * inverse;
        for (int s = 24; s <= 25; ++s)
            for (int d = -12; d <= 12; ++d) {
                if (d == 0 || d % (int)(1u << (twos < 5 ? twos : 5)) != 0) continue;
                const int dd = d / (int)(1u << twos); /* exact: twos <= 3 here */
                const uint32_t modulus = 1u << (s - twos);
                for (uint64_t M = (0u - (uint32_t)dd * inverse) & (modulus - 1u); M < (1u << 25); M += modulus) {
                    if (M < (1u << 24) || !(M & 1u)) continue;
                    const uint64_t t = M * B + (uint64_t)(int64_t)d, ia = t >> s;
                    if ((t & ((1ull << s) - 1ull)) != 0) return 2;
                    if (ia < (1u << 23) || ia >= (1u << 24) || (s == 24) != (ia >= B)) continue;
                    const float a = (float)ia, q = a * y, r = fmaf(-b, q, a);
                    ++cases;
                    wrong += fmaf(r, y, q) != a / b;
                }
            }
    }
    printf("%ld %ld\n", cases, wrong);
    return 0;
}
