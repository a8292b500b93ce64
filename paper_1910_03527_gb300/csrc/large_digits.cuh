#pragma once
// The float64 sigma of one large space on the tensor cores (large_digits.cu).
#include "common.cuh"
#include "digits.cuh"

namespace mbe {

constexpr int DIGITS_EXP = 450;  // largest |exponent| of an operand's scale

struct DigitsArgs {
    int P, Ns, R, nsp;    // nsp: Ns rounded up to 64, the row stride of planes and inv
    int n;                // orbitals, if c may have any spread (see k_digits_near), else 0
    const int32_t *tab;   // [Ns][R] replacement lists
    const int32_t *tabT;  // [R][Ns]
    int32_t *inv;         // [P][nsp] K << 1 | neg, or -1
    const double *V;      // [P][P]
    const double *hd;     // [Ns] diagonal of Hs
    const double *c;      // [Ns][Ns]
    uint16_t *planes;     // [DIGITS][Ns][nsp] digits of c (scratch)
    unsigned long long *maxb;  // [4] bits of the largest |V|, |off-diagonal Hs| and |c|; not 0: digits are not used
    uint16_t *hplanes;  // [DIGITS][Ns][nsp] digits of Hs without its diagonal
    double *sigma;        // [Ns][Ns], written
};

// Strings per chunk of c with which a space's operands fit in shared memory (0: not at all).
int large_digits_chunk(size_t smem_optin, int P, int Ns, int R);
// Per space: hd, Hs's planes, inv and the maxima of V and Hs (a's pointers to them are written).
int large_digits_setup(cudaStream_t st, int sm_count, const DigitsArgs &a, const double *Hs, double *hd);
// sigma = H c, all terms; returns at once on values that digits_usable() leaves to float64.
int large_sigma_digits(cudaStream_t st, int sm_count, size_t smem_optin, const DigitsArgs &a, int chunk);

// 2^e (e within the normal range)
__device__ inline double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// Exponent E of the power of two above a largest absolute value, from its bits.
__device__ inline int bits_exponent(unsigned long long b)
{
    const int E = (int)(b >> 52) - 1022;
    return E < -DIGITS_EXP ? -DIGITS_EXP : E;
}

// Whether the scales of all operands are far from the ends of float64's range (an infinity or a
// NaN has the largest exponent); zero operands are.
__device__ inline bool digits_in_range(const unsigned long long *maxb)
{
    for (int i = 0; i < 3; ++i) {
        const int E = (int)(maxb[i] >> 52) - 1022;
        if (maxb[i] != 0ull && (E < -DIGITS_EXP || E > DIGITS_EXP)) return false;
    }
    return true;
}

// ... and they are not too uneven either (k_digits_even).
__device__ inline bool digits_usable(const unsigned long long *maxb) { return maxb[3] == 0ull && digits_in_range(maxb); }

// Largest of the lanes' |v|, as bits (in which a NaN is above all numbers), into *out.
__device__ inline void max_bits(unsigned long long b, unsigned long long *out)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, b, o);
        b = u > b ? u : b;
    }
    if ((threadIdx.x & 31) == 0 && b != 0ull) atomicMax(out, b);
}

}  // namespace mbe
