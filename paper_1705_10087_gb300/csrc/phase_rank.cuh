// Device pieces shared by the visits of a 1-D segment (phase_reg_impl.cuh) and of a
// 2-D tile (csc2d_tile.cuh): keys of the argmax, the ranking of a staged column
// (the atoms of one position) and background copies of neighbours' columns.
#pragma once

#include "csc_internal.cuh"
#include "packed.cuh"

namespace csc {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kActive = 128;   // listed coordinates of a visit at most

// x, hidden from the optimiser: keeps multiples of a stride from being hoisted
// out of the update loop into registers.
__device__ __forceinline__ int64_t opaque(int64_t x)
{
    asm volatile("" : "+l"(x));
    return x;
}
__device__ __forceinline__ int opaque(int x)
{
    asm volatile("" : "+r"(x));
    return x;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned hi, unsigned lo)
{
    const unsigned hmax = __reduce_max_sync(kFull, hi);
    const unsigned lmax = __reduce_max_sync(kFull, hi == hmax ? lo : 0u);
    return ((unsigned long long)hmax << 32) | lmax;
}

// Index word of a key, complemented so that the largest key is the lowest
// (atom, position): k << shift | pos | listed << 1 | sign of dZ, where pos holds
// the position in the tile in bits 2 .. shift - 1, in the order of ties.
__device__ __forceinline__ unsigned key_index(unsigned k, int shift, unsigned pos, unsigned listed,
                                              unsigned neg)
{
    return ~((k << shift) | pos | (listed << 1) | neg);
}

// A column's r (atom rows src + i ld, n of them) copied to shared memory in the
// background (cp.async, completed by halo_wait in the same thread).
template <int N>
__device__ __forceinline__ void halo_load(unsigned long long *dst, const float *src, int64_t ld,
                                          int n)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int64_t step = opaque(ld);
#pragma unroll
    for (int i = 0; i < N; i++, src += step)
        if (i < n)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * i),
                         "l"(__cvta_generic_to_global(src))
                         : "memory");
}
template <int N>
__device__ __forceinline__ void halo_store(const unsigned long long *src, float *dst, int64_t ld,
                                           int n)
{
    const int64_t step = opaque(ld);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        float lo, hi;
        unpack2(src[i / 2], lo, hi);
        if (i < n)
            *dst = lo;
        dst += step;
        if (i + 1 < n)
            *dst = hi;
        dst += step;
    }
}
__device__ __forceinline__ void halo_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// v = (|r| - lam) / n of the two atoms of a pair (rn: 1 / n)
__device__ __forceinline__ void excess2(unsigned long long r, unsigned long long rn, float lam,
                                        float &v0, float &v1)
{
    float a, b;
    unpack2(r, a, b);
    unpack2(mul2(pack2(fabsf(a) - lam, fabsf(b) - lam), rn), v0, v1);
}

// The best of one column's atoms with z == 0 from v[i] = (|r_i| - lambda) / n_i
// (NaN for atoms on the active list): its key, 0 when nothing moves.  r: the
// staged column.  coord_step's float32 resolution floor can reject the best
// only when its excess over lambda is a few ulps; then all are tested (but for
// those of the mask unl: nonzero and not listed, v[i] < 0).
template <int N>
__device__ __forceinline__ void rank_column(const float (&v)[N], const float *r, const float *rn,
                                            float lam, unsigned unl, unsigned kbase, int shift,
                                            unsigned pos, unsigned &khi, unsigned &klo)
{
    constexpr float kFloor = 4.76837158203125e-07f;  // 2^-21
    // (four chains, so that their latencies overlap)
    float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        float &x = m[(i >> 1) & 3];
        x = fmaxf(x, fmaxf(v[i], v[i + 1]));
    }
    float vm = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
    khi = 0u;
    klo = 0u;
    if (vm > 0.f) {
        // the first atom that attains it
        int b[2] = {N, N};
#pragma unroll
        for (int i = N / 2 - 1; i >= 0; i--) {
            if (v[i] == vm)
                b[0] = i;
            if (v[i + N / 2] == vm)
                b[1] = i + N / 2;
        }
        int bi = min(b[0], b[1]);
        float rs = r[bi];
        if (vm < fabsf(rs) * kFloor * rn[bi]) {
            vm = 0.f;
#pragma unroll 1
            for (int i = 0; i < N; i++) {
                const float y = r[i], x = (fabsf(y) - lam) * rn[i];
                if (!(unl >> i & 1u) && x > vm && !(x < fabsf(y) * kFloor * rn[i])) {
                    vm = x;
                    bi = i;
                    rs = y;
                }
            }
        }
        if (vm > 0.f) {
            khi = __float_as_uint(vm);
            klo = key_index(kbase + bi, shift, pos, 0u, __float_as_uint(rs) >> 31);
        }
    }
}

// Adds the coordinates of a column whose Z is nonzero but not listed (bits of
// zm) to its key (khi, klo); r: the staged column, zcol + i ld: Z of atom kbase + i.
__device__ __forceinline__ void rank_unlisted(unsigned zm, const float *r, const float *zcol,
                                              int64_t ld, const float *nrm, const float *rn,
                                              float lam, unsigned kbase, int shift, unsigned pos,
                                              unsigned &khi, unsigned &klo)
{
#pragma unroll 1
    for (; zm; zm &= zm - 1) {
        const int i = __ffs((int)zm) - 1;
        float zn, d;
        coord_step(r[i], zcol[(int64_t)i * ld], nrm[i], rn[i], lam, &zn, &d);
        const unsigned h = __float_as_uint(fabsf(d));
        const unsigned l = key_index(kbase + i, shift, pos, 0u, d < 0.f ? 1u : 0u);
        if (fabsf(d) > 0.f && (h > khi || (h == khi && l > klo))) {
            khi = h;
            klo = l;
        }
    }
}

}  // namespace csc
