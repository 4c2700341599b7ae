// Arithmetic modulo one prime on the device (series and Chinese remaindering).
#pragma once

#include <stdint.h>

namespace cp {

// Arithmetic modulo a prime p < 2^31.  Products use Barrett reduction with
// m = floor((2^64 - 1) / p): q = floor(x m / 2^64) undershoots floor(x / p) by at
// most 2 for x < 2^62, so x - q p < 3p needs at most two subtractions.
struct Mod {
    uint32_t p;
    uint64_t m;
};
__device__ __forceinline__ Mod make_mod(uint32_t p) { return Mod{p, 0xFFFFFFFFFFFFFFFFull / p}; }
__device__ __forceinline__ uint32_t mm(uint32_t a, uint32_t b, const Mod &M) {
    const uint64_t x = (uint64_t)a * b;
    uint64_t r = x - __umul64hi(x, M.m) * M.p;
    if (r >= M.p) r -= M.p;
    if (r >= M.p) r -= M.p;
    return (uint32_t)r;
}
__device__ __forceinline__ uint32_t ad(uint32_t a, uint32_t b, uint32_t p) {
    uint32_t t = a + b;
    return t >= p ? t - p : t;
}
__device__ __forceinline__ uint32_t sb(uint32_t a, uint32_t b, uint32_t p) { return a >= b ? a - b : a + p - b; }
__device__ __forceinline__ uint32_t from_int(long long v, uint32_t p) {
    long long r = v % (long long)p;
    return (uint32_t)(r < 0 ? r + p : r);
}
__device__ __forceinline__ uint32_t pw(uint32_t a, uint32_t e, const Mod &M) {
    uint32_t r = 1;
    while (e) {
        if (e & 1) r = mm(r, a, M);
        a = mm(a, a, M);
        e >>= 1;
    }
    return r;
}

}  // namespace cp
