// The phase kernel with thread-private r: the block form of a segment's visit.
//
// A visit applies a serial chain of updates (argmax -> coefficients -> window
// update -> re-evaluation), so what bounds it is the latency of one link and,
// with several blocks on an SM, the instructions and shared-memory traffic of
// one link.  The coordinates of a segment are split between two kinds of warps:
//   column threads  thread (c, g) owns the columns jj == c (mod cb) and, of
//     each, the NQ float4 groups of atoms [g NQ, (g+1) NQ), z == 0 only.  Their r
//     is staged in shared memory, a column's atoms one after the other (odd
//     stride in quads: 128-bit accesses without bank conflicts).  A column is
//     ranked with straight-line code: |Delta Z| = (|r| - lambda) / n of all its
//     atoms.
//   the active warp  one lane per coordinate with z != 0 (and those that became
//     nonzero in this visit): r and z of the lane's coordinates, updated with
//     one coefficient each and ranked with the full coordinate step.  A segment
//     has a few tens of them; walked by the column threads, their case
//     distinctions cost every warp more instructions than the z == 0 atoms.
// A column entry whose coordinate is on the active list holds NaN, which no
// maximum picks.  A coordinate that wins with z == 0 moves to the list: it is at
// its optimum then (its next |Delta Z| is below the float32 floor), so the list
// needs it only from the next update on.  Beyond kActive entries coordinates
// stay with their column thread, which ranks them one by one from Z in global
// memory.
// The idle neighbours' columns within L-1 of the segment (no other block of the
// launch touches them) are fetched to shared memory in the background, updated
// there and written back once: atomic additions to global memory, 25 in a row
// per thread, took 900 to 3600 of the 2900 to 5700 cycles of a link.
//
// Arithmetic, order of the updates and ties are those of visit_segment in
// kernel_phase.cu (which still runs the segments this form does not hold): the
// same key order (|Delta Z|, then the lowest atom, then the lowest column), the
// same coordinate step, the same float operations per coordinate.
//
// cb >= 2L-1, so the window's columns go to distinct threads of a group; the
// groups of a column share an update by atoms and meet only in the argmax.
//
// Measured against visit_segment (summed phase launches of one solve):
//   P=7, K=25, L=64, T=200,000, 1024 segments   722 -> 518 us
//   P=5, K=18, L=51, T=60,013                   2737 -> 580 us
//   P=1, K=5, L=16, T=2000, 10 segments         734 -> 328 us
//   P=1, K=25, L=200, T=5,000,000               26.8 -> 22.1 ms
// What bounds it now: 2300 cycles per link with one block on an SM (the L2 round
// trip of the coefficients 600-700 of them); with five blocks the L1/shared
// pipe (76% busy).
#pragma once

#include "csc_internal.cuh"
#include "phase_reg.cuh"

namespace csc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRegWarps = 16;  // column warps of a block at most (and one active warp)
constexpr int kRegAtoms = 32 * kRegWarps;  // padded atoms: at most 16 groups of 8 float4
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
// (atom, column): k << 17 | slot << 12 | class << 2 | listed << 1 | sign of dZ.
__device__ __forceinline__ unsigned key_index(unsigned k, unsigned pos, unsigned listed,
                                              unsigned neg)
{
    return ~((k << 17) | pos | (listed << 1) | neg);
}
__device__ __forceinline__ unsigned key_pos(unsigned slot, unsigned c)
{
    return (slot << 12) | (c << 2);
}

// Packed pairs of floats (one 64-bit register pair, two operations at once).
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long x;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(lo), "f"(hi));
    return x;
}
__device__ __forceinline__ void unpack2(unsigned long long x, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    // (scalar: the packed sum of a packed product would be contracted)
    float a0, a1, b0, b1;
    unpack2(a, a0, a1);
    unpack2(b, b0, b1);
    return pack2(__fadd_rn(a0, b0), __fadd_rn(a1, b1));
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
// only when its excess over lambda is a few ulps; then all are tested.
template <int N>
__device__ __forceinline__ void rank_column(const float (&v)[N], const float *r, const float *rn,
                                            float lam, unsigned kbase, unsigned pos,
                                            unsigned &khi, unsigned &klo)
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
                if (x > vm && !(x < fabsf(y) * kFloor * rn[i])) {
                    vm = x;
                    bi = i;
                    rs = y;
                }
            }
        }
        if (vm > 0.f) {
            khi = __float_as_uint(vm);
            klo = key_index(kbase + bi, pos, 0u, __float_as_uint(rs) >> 31);
        }
    }
}

// Adds the coordinates of a column whose Z is nonzero but not listed (bits of
// zm) to its key (khi, klo); r: the staged column, zcol + i ld: Z of atom kbase + i.
__device__ __forceinline__ void rank_unlisted(unsigned zm, const float *r, const float *zcol,
                                              int64_t ld, const float *nrm, const float *rn,
                                              float lam,
                                              unsigned kbase, unsigned pos, unsigned &khi,
                                              unsigned &klo)
{
#pragma unroll 1
    for (; zm; zm &= zm - 1) {
        const int i = __ffs((int)zm) - 1;
        float zn, d;
        coord_step(r[i], zcol[(int64_t)i * ld], nrm[i], rn[i], lam, &zn, &d);
        const unsigned h = __float_as_uint(fabsf(d));
        const unsigned l = key_index(kbase + i, pos, 0u, d < 0.f ? 1u : 0u);
        if (fabsf(d) > 0.f && (h > khi || (h == khi && l > klo))) {
            khi = h;
            klo = l;
        }
    }
}

// One launch of a phase.  drain == 0: block b visits segment phase_list[b];
// else the blocks drain the queue (see launch_phase_drain).
// TAIL: the last group of atoms may hold fewer than NQ quads.
template <int NQ, bool TAIL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    phase_reg_kernel(PhaseParams pp, int cb, int drain)
{
    constexpr int N = 4 * NQ;
    const float kNan = __int_as_float(0x7fffffff);
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ __align__(16) unsigned long long s_key[2][32];
    __shared__ __align__(16) float s_nrm[kRegAtoms], s_rn[kRegAtoms];
    // active list: r, z, index word of the key (flags 0), Z' of the last step
    __shared__ __align__(16) float4 s_act[kActive];
    __shared__ double s_dec[kRegWarps + 1];
    __shared__ int s_go, s_idx, s_nact;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int nt = blockDim.x - 32;  // column threads; the last warp has the active list
    const bool is_col = tid < nt;
    const int K = pp.K, L = pp.L, W2 = 2 * L - 1, KQ = pp.Kp >> 2;
    const int grp = tid / cb, c = tid - grp * cb;  // (cb is a multiple of 32)
    const int q0 = grp * NQ;
    const unsigned kbase = is_col ? 4u * (unsigned)q0 : 0u;
    const int quads = KQ - q0 < NQ ? KQ - q0 : NQ;  // of this thread (TAIL)
    const int gi = pp.g_dev ? *pp.g_dev + pp.g : pp.g;
    const int g_round = pp.g_round_dev ? *pp.g_round_dev : pp.g_round;
    const float *const nrm = s_nrm + kbase, *const rn = s_rn + kbase;
    // columns of this thread's group of atoms: own ones at jj, after them the
    // halo, left ones at h = jj + L-1, right ones at h = L-1 + jj - w
    constexpr int kStride = (NQ | 1) * 2;  // pairs of a column
    const int groups = nt / cb, g = is_col ? grp : 0, w_max = pp.w_max;
    unsigned long long *const all = reinterpret_cast<unsigned long long *>(dyn);
    unsigned long long *const rs = all + g * (w_max + 2 * L - 2) * kStride;
    unsigned long long *const halo = rs + w_max * kStride;
    unsigned long long *const keys = all + groups * (w_max + 2 * L - 2) * kStride;
    unsigned long long *const skey = keys + g * w_max;
    unsigned *const slst = reinterpret_cast<unsigned *>(keys + groups * w_max) + g * w_max;
    unsigned *const sunl = slst + groups * w_max;

    for (int k = tid; k < 4 * NQ * groups; k += blockDim.x) {
        // (rn = 0 beyond the last atom: no excess there)
        const float n = k < K ? pp.norms[k] : 1.f;
        s_nrm[k] = n;
        s_rn[k] = k < K ? __frcp_rn(n) : 0.f;
    }
    if (tid < 64)
        s_key[tid >> 5][tid & 31] = 0ull;

    // a full sweep (the previous c launches of this round) applied nothing
    auto sweep_idle = [&]() {
        long long sum = 0;
#pragma unroll 1
        for (int j = gi - pp.c; j < gi; j++)
            sum += *(volatile long long *)&pp.upd[j & (kPhaseRing - 1)];
        return sum == 0;
    };
    const int qn = drain ? *pp.qlen : 1;
    // an empty queue visits nothing, so the test made at the start of every
    // visit is also made here once
    if (drain && blockIdx.x == 0 && tid == 0 && gi - g_round >= pp.c &&
        !*(volatile int *)pp.done && sweep_idle())
        *(volatile int *)pp.done = gi + 1;

    for (;;) {
        int m;
        if (drain) {
            if (tid == 0)
                s_idx = atomicAdd(pp.qhead, 1);
            __syncthreads();
            const int idx = s_idx;
            if (idx >= qn)
                return;
            m = pp.queue[idx];
        } else {
            m = pp.phase_list[blockIdx.x];
        }
        // early exits, decided by one thread so the block stays uniform (total
        // is being incremented by other blocks of this launch); the segment's
        // description is read by all meanwhile
        if (tid == 0) {
            const int done = *(volatile int *)pp.done;
            const long long total = *(volatile long long *)pp.total;
            const unsigned char dirty = *(volatile unsigned char *)&pp.dirty[m];
            int go = !done && total < pp.max_updates;
            if (go && gi - g_round >= pp.c && sweep_idle()) {
                *(volatile int *)pp.done = gi + 1;  // same value from every block
                go = 0;
            }
            s_go = go && dirty;
            s_nact = 0;
        }
        const SigDesc *sdp = pp.sig + pp.seg_sig[m];
        const int64_t s0 = pp.seg_s[m];
        const int w = (int)(pp.seg_e[m] - s0);
        const int64_t ld = sdp->ld;
        // this thread's atoms at the segment's first column
        float *const rbase = sdp->r + (int64_t)kbase * ld + s0;
        float *const zbase = sdp->Z + (int64_t)kbase * ld + s0;
        __builtin_assume(__isGlobal(rbase));
        __builtin_assume(__isGlobal(zbase));
        // valid columns of the problem, relative to the segment (w < 2^16)
        const int lo_valid = s0 < kMaxL ? -(int)s0 : -kMaxL;
        const int hi_valid = sdp->Tz - s0 < (1 << 20) ? (int)(sdp->Tz - s0) : 1 << 20;
        const float lam = sdp->lam, tol = sdp->tol;
        __syncthreads();
        if (!s_go) {
            if (!drain)
                return;
            __syncthreads();  // s_go and s_idx are rewritten by the next visit
            continue;
        }

        // ---- the thread's columns: r, nonzeros of Z listed, best coordinate --
        unsigned khi = 0, klo = 0;  // of an active lane: its best key
        // own slots (bit s) and halo columns whose r changed in this visit
        unsigned changed = 0;
        constexpr unsigned kLeft = 1u << 31, kRight = 1u << 30;
        // the columns of this class within L-1 of the segment on either side (idle
        // neighbours' columns, which no other block of the launch touches):
        // their r on its way to shared memory meanwhile
        const int jl = c - cb, jr = w <= c ? c : c + (w - c + cb - 1) / cb * cb;
        const bool has_l = is_col && jl >= 1 - L && jl >= lo_valid;
        const bool has_r = is_col && jr < w + L - 1 && jr < hi_valid;
        if (has_l)
            halo_load<N>(halo + (jl + L - 1) * kStride, rbase + jl, ld, K - (int)kbase);
        if (has_r)
            halo_load<N>(halo + (L - 1 + jr - w) * kStride, rbase + jr, ld, K - (int)kbase);
        if (is_col)
#pragma unroll 1
            for (int s = 0, jj = c; jj < w; s++, jj += cb) {
                const int64_t step = opaque(ld);
                const unsigned pos = key_pos((unsigned)s, (unsigned)c);
                unsigned zb = 0, zl = 0;
                {
                    const float *zp = zbase + jj;
#pragma unroll
                    for (int i = 0; i < N; i++, zp += step)
                        zb |= ((int)kbase + i < K && *zp != 0.f ? 1u : 0u) << i;
                }
#pragma unroll 1
                for (unsigned rest = zb; rest; rest &= rest - 1) {
                    const int i = __ffs((int)rest) - 1, a = atomicAdd(&s_nact, 1);
                    if (a < kActive) {
                        const int64_t o = (int64_t)i * step + jj;
                        s_act[a] = make_float4(rbase[o], zbase[o],
                                               __uint_as_float(((kbase + i) << 17) | pos), 0.f);
                        zl |= 1u << i;
                    }
                }
                zb &= ~zl;
                float v[N];
                {
                    const float *rp = rbase + jj;
#pragma unroll
                    for (int i = 0; i < N; i++, rp += step)
                        v[i] = (int)kbase + i < K ? *rp : 0.f;
                }
#pragma unroll
                for (int i = 0; i < N; i++)
                    if (zl >> i & 1u)
                        v[i] = kNan;
                unsigned long long *const col = rs + jj * kStride;
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    const ulonglong2 n4 = *reinterpret_cast<const ulonglong2 *>(rn + 4 * q);
                    const ulonglong2 x = make_ulonglong2(pack2(v[4 * q], v[4 * q + 1]),
                                                         pack2(v[4 * q + 2], v[4 * q + 3]));
                    *reinterpret_cast<ulonglong2 *>(col + 2 * q) = x;
                    excess2(x.x, n4.x, lam, v[4 * q], v[4 * q + 1]);
                    excess2(x.y, n4.y, lam, v[4 * q + 2], v[4 * q + 3]);
                }
                if (zb) {
#pragma unroll
                    for (int i = 0; i < N; i++)
                        if (zb >> i & 1u)
                            v[i] = -1.f;
                }
                const float *const rc = reinterpret_cast<const float *>(col);
                rank_column<N>(v, rc, rn, lam, kbase, pos, khi, klo);
                if (zb)
                    rank_unlisted(zb, rc, zbase + jj, ld, nrm, rn, lam, kbase, pos, khi, klo);
                skey[jj] = ((unsigned long long)khi << 32) | klo;
                slst[jj] = zl;
                sunl[jj] = zb;
            }
        __syncthreads();
        int nact = s_nact < kActive ? s_nact : kActive;
        float decrease = 0.f;  // this thread's updates of the visit (at most u terms)

        // the lane's listed coordinates after the update (k0, column jw, dZ) of
        // key index word win (none of them with upd = false), two at a time; leaves
        // the lane's best key in khi, klo
        auto active_step = [&](bool upd, unsigned win, int k0, int jw, float delta) {
            khi = klo = 0u;
            const float *const C1 = pp.Ct;
#pragma unroll 1
            for (int a0 = lane; a0 < nact; a0 += 64) {
                float4 e[2];
                float cv[2];
                bool in[2];
#pragma unroll
                for (int x = 0; x < 2; x++) {
                    const int a = a0 + 32 * x;
                    in[x] = a < nact;
                    e[x] = in[x] ? s_act[a] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const unsigned id = __float_as_uint(e[x].z);
                    const int jj = (int)(id >> 12 & 31u) * cb + (int)(id >> 2 & 0x3ffu);
                    const int k = (int)(id >> 17), d = jj - jw + (L - 1);
                    cv[x] = 0.f;
                    if (upd && in[x] && d >= 0 && d < W2)
                        cv[x] = __ldg(C1 + (((k0 * KQ + (k >> 2)) * W2 + d) << 2) + (k & 3));
                }
#pragma unroll
                for (int x = 0; x < 2; x++) {
                    if (!in[x])
                        continue;
                    const unsigned id = __float_as_uint(e[x].z);
                    const unsigned k = id >> 17;
                    const float n = s_nrm[k];
                    if (upd && (id | 2u) == (win & ~1u)) {
                        // Prop. A.1 from r before this update touches it:
                        // dZ (r - n dZ / 2) + lam (|z| - |u|)
                        const float u = e[x].w, z = u - delta;
                        decrease +=
                            delta * (e[x].x - 0.5f * n * delta) + lam * (fabsf(z) - fabsf(u));
                        e[x].y = u;
                        zbase[(int64_t)k * ld + jw] = u;
                    }
                    if (upd)
                        e[x].x = fmaf(-cv[x], delta, e[x].x);
                    float zn, d;
                    coord_step(e[x].x, e[x].y, n, s_rn[k], lam, &zn, &d);
                    e[x].w = zn;
                    s_act[a0 + 32 * x] = e[x];
                    const unsigned h = __float_as_uint(fabsf(d));
                    const unsigned l = ~(id | 2u | (d < 0.f ? 1u : 0u));
                    if (fabsf(d) > 0.f && (h > khi || (h == khi && l > klo))) {
                        khi = h;
                        klo = l;
                    }
                }
            }
        };
        if (!is_col)
            active_step(false, 0u, 0, 0, 0.f);

        const char *const Ctb = reinterpret_cast<const char *>(pp.Ct);
        const unsigned cstep = (unsigned)W2 * 16u;
        int nupd = 0;
        int jmin = w, jmax = -1;
        bool capped = false;
#pragma unroll 1
        for (int it = 0;; it++) {
            // ---- block argmax of the keys --------------------------------
            unsigned mh = khi, ml = klo;
            // (a single own column's key is still in khi, klo)
            if (is_col && w > cb) {
                unsigned long long my = 0ull;
#pragma unroll 1
                for (int jj = c; jj < w; jj += cb) {
                    const unsigned long long x = skey[jj];
                    my = x > my ? x : my;
                }
                mh = (unsigned)(my >> 32);
                ml = (unsigned)my;
            }
            unsigned long long best = warp_max_u64(mh, ml);
            if (lane == 0)
                s_key[it & 1][warp] = best;
            __syncthreads();
            if (nwarps <= 6) {
                const ulonglong2 *const k2 = reinterpret_cast<const ulonglong2 *>(s_key[it & 1]);
                const ulonglong2 x = k2[0], y = k2[1], z = k2[2];
                const unsigned long long p = x.x > x.y ? x.x : x.y, q = y.x > y.y ? y.x : y.y,
                                         r = z.x > z.y ? z.x : z.y, o = p > q ? p : q;
                best = o > r ? o : r;
            } else {
                const unsigned long long x = s_key[it & 1][lane];
                best = warp_max_u64((unsigned)(x >> 32), (unsigned)x);
            }
            // (kept in ordinary registers: the decode is a chain, and the uniform
            // unit's latency is longer)
            best = (unsigned long long)opaque((int64_t)best);
            const float adz = __uint_as_float((unsigned)(best >> 32));
            if (!(adz >= tol))
                break;
            if (nupd >= pp.u) {
                capped = true;
                break;
            }
            // the winner and dZ = +-|dZ| from its key
            const unsigned flat = ~(unsigned)best;
            const int k0 = (int)(flat >> 17), sw = (int)(flat >> 12 & 31u),
                      cw = (int)(flat >> 2 & 0x3ffu);
            const bool listed = flat & 2u;
            const float delta = (flat & 1u) ? -adz : adz;
            const unsigned long long ndelta = pack2(-delta, -delta);
            const int jw = cw + sw * cb;
            // a winner from a column is listed from the next update on
            const int slot_new = nact;
            const bool to_list = !listed && nact < kActive;

            // ---- Eq. beta_up (r form) on the window ----------------------
            if (!is_col) {
                active_step(true, flat, k0, jw, delta);
            } else {
                // window position of this thread: c - (cw - (L-1)) mod cb, in
                // the winner's column slot or a neighbouring one
                int off = c + (L - 1) - cw;
                const int ds = off < 0 ? 1 : (off >= cb ? -1 : 0);
                off += ds * cb;
                const int jj = jw - (L - 1) + off;
                if (off < W2 && jj >= lo_valid && jj < hi_valid) {
                    // coefficients S_{k,k0}[t-t0]: float4 group q of (k0, lag) at
                    // Ct4[(k0 * KQ + q) * W2 + lag] (consecutive lags adjacent; a
                    // group beyond the last repeats it: its atoms have rn = 0)
                    unsigned long long cv[2 * NQ];
                    {
                        unsigned o = (unsigned)((k0 * KQ + q0) * W2 + off) * 16u;
#pragma unroll
                        for (int q = 0; q < NQ; q++) {
                            const ulonglong2 y =
                                __ldg(reinterpret_cast<const ulonglong2 *>(Ctb + o));
                            cv[2 * q] = y.x;
                            cv[2 * q + 1] = y.y;
                            if (!TAIL || q + 1 < quads)
                                o += cstep;
                        }
                    }
                    if (jj >= 0 && jj < w) {
                        const int s = sw + ds;
                        unsigned long long *const col = rs + jj * kStride;
                        float *const rc = reinterpret_cast<float *>(col);
                        // (none is unlisted while the list has room)
                        unsigned zb = nact < kActive ? 0u : sunl[jj];
                        const unsigned pos = key_pos((unsigned)s, (unsigned)c);
                        if (jj == jw && !listed && (k0 >> 2) >= q0 && (k0 >> 2) < q0 + NQ) {
                            const int i0 = k0 - (int)kbase;
                            const unsigned bit = 1u << i0;
                            const float n = nrm[i0], r0 = rc[i0];
                            float *const zp = zbase + (int64_t)i0 * opaque(ld) + jj;
                            float u = delta, z = 0.f;
                            if (to_list) {
                                s_act[slot_new] = make_float4(
                                    fmaf(-n, delta, r0), u,
                                    __uint_as_float(((unsigned)k0 << 17) | pos), u);
                                slst[jj] |= bit;
                                rc[i0] = kNan;
                            } else {
                                // the list is full: Z' as the key's step found it
                                float d;
                                coord_step(r0, zb & bit ? *zp : 0.f, n, rn[i0], lam, &u, &d);
                                z = u - delta;
                                zb = u != 0.f ? (zb | bit) : (zb & ~bit);
                                sunl[jj] = zb;
                            }
                            // Prop. A.1 from r before this update touches it:
                            // dZ (r - n dZ / 2) + lam (|z| - |u|)
                            decrease +=
                                delta * (r0 - 0.5f * n * delta) + lam * (fabsf(z) - fabsf(u));
                            *zp = u;
                        }
                        float v[N];
#pragma unroll
                        for (int q = 0; q < NQ; q++) {
                            const ulonglong2 n4 = *reinterpret_cast<const ulonglong2 *>(rn + 4 * q);
                            ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(col + 2 * q);
                            x.x = fma2(cv[2 * q], ndelta, x.x);
                            x.y = fma2(cv[2 * q + 1], ndelta, x.y);
                            *reinterpret_cast<ulonglong2 *>(col + 2 * q) = x;
                            excess2(x.x, n4.x, lam, v[4 * q], v[4 * q + 1]);
                            excess2(x.y, n4.y, lam, v[4 * q + 2], v[4 * q + 3]);
                        }
                        changed |= 1u << s;
                        if (zb) {
#pragma unroll
                            for (int i = 0; i < N; i++)
                                if (zb >> i & 1u)
                                    v[i] = -1.f;
                        }
                        rank_column<N>(v, rc, rn, lam, kbase, pos, khi, klo);
                        if (zb)
                            rank_unlisted(zb, rc, zbase + jj, ld, nrm, rn, lam, kbase, pos, khi,
                                          klo);
                        skey[jj] = ((unsigned long long)khi << 32) | klo;
                    } else {
                        // an idle neighbour's column: its r, product and sum
                        // rounded one after the other (as by an atomic addition)
                        halo_wait();
                        const int h = jj < 0 ? jj + L - 1 : L - 1 + jj - w;
                        ulonglong2 *const col = reinterpret_cast<ulonglong2 *>(halo + h * kStride);
#pragma unroll
                        for (int q = 0; q < NQ; q++) {
                            ulonglong2 x = col[q];
                            x.x = add2(x.x, mul2(cv[2 * q], ndelta));
                            x.y = add2(x.y, mul2(cv[2 * q + 1], ndelta));
                            col[q] = x;
                        }
                        changed |= jj < 0 ? kLeft : kRight;
                    }
                }
            }
            nact += to_list ? 1 : 0;
            nupd++;
            jmin = jw < jmin ? jw : jmin;
            jmax = jw > jmax ? jw : jmax;
        }

        // ---- write back, spill bookkeeping, trace -----------------------
        // (Z went to global memory when it was applied)
        halo_wait();  // (nothing is in flight when the next visit or the end comes)
        if (is_col) {
            if (changed & kLeft)
                halo_store<N>(halo + (jl + L - 1) * kStride, rbase + jl, ld, K - (int)kbase);
            if (changed & kRight)
                halo_store<N>(halo + (L - 1 + jr - w) * kStride, rbase + jr, ld, K - (int)kbase);
#pragma unroll 1
            for (int s = 0, jj = c; jj < w; s++, jj += cb)
                if (changed >> s & 1u) {
                    const unsigned skip = slst[jj];
                    float *rdst = rbase + jj;
                    const int64_t step = opaque(ld);
#pragma unroll
                    for (int i = 0; i < N; i += 2) {
                        float lo, hi;
                        unpack2(rs[jj * kStride + i / 2], lo, hi);
                        if ((int)kbase + i < K && !(skip >> i & 1u))
                            *rdst = lo;
                        rdst += step;
                        if ((int)kbase + i + 1 < K && !(skip >> (i + 1) & 1u))
                            *rdst = hi;
                        rdst += step;
                    }
                }
        } else if (nupd > 0) {
#pragma unroll 1
            for (int a = lane; a < nact; a += 32) {
                const float4 e = s_act[a];
                const unsigned id = __float_as_uint(e.z);
                const int jj = (int)(id >> 12 & 31u) * cb + (int)(id >> 2 & 0x3ffu);
                rbase[(int64_t)(id >> 17) * ld + jj] = e.x;
            }
        }
        for (int o = 16; o > 0; o >>= 1)
            decrease += __shfl_xor_sync(kFull, decrease, o);
        if (lane == 0)
            s_dec[warp] = (double)decrease;
        __syncthreads();
        if (tid == 0) {
            double dsum = 0.0;
#pragma unroll 1
            for (int i = 0; i < nwarps; i++)
                dsum += s_dec[i];
            pp.dirty[m] = capped ? 1 : 0;
            if (nupd > 0) {
                // neighbours whose r changed: segments meeting [tmin-L+1, tmax+L-1];
                // they and this segment are also touched: r changed there
                const int64_t lo = s0 + jmin - (L - 1), hi = s0 + jmax + (L - 1);
                const int seg_lo = sdp->seg0, seg_hi = seg_lo + sdp->nseg;
#pragma unroll 1
                for (int mm = m - 1; mm >= seg_lo && pp.seg_e[mm] > lo; mm--) {
                    pp.dirty[mm] = 1;
                    pp.touched[mm] = 1;
                }
#pragma unroll 1
                for (int mm = m + 1; mm < seg_hi && pp.seg_s[mm] <= hi; mm++) {
                    pp.dirty[mm] = 1;
                    pp.touched[mm] = 1;
                }
                pp.touched[m] = 1;
                const int slot = gi & (kPhaseRing - 1);
                atomicAdd(reinterpret_cast<unsigned long long *>(&pp.upd[slot]),
                          (unsigned long long)nupd);
                atomicAdd(reinterpret_cast<unsigned long long *>(pp.total),
                          (unsigned long long)nupd);
                atomicAdd(reinterpret_cast<unsigned long long *>(pp.visits), 1ull);
                atomicAdd(&pp.dec[slot], dsum);
                atomicMax(&pp.tend[slot], globaltimer_ns());
            }
        }
        if (!drain)
            return;
        // the next visit rewrites the shared state read above
        __syncthreads();
    }
}

// The instantiation for blocks of `block` threads (registers: at most 65536 /
// (threads x blocks per SM)).  dense: more segments than fit at once, so the
// blocks per SM count; else a segment's chain of
// updates counts.  One group of atoms (K <= 32) has a form for every NQ, so no
// quad is padding; with more groups the last one may be short (TAIL).
template <int NQ, bool TAIL>
RegKernel by_block(int block, bool dense)
{
    if (block <= 160)
        return dense ? phase_reg_kernel<NQ, TAIL, 160, 5> : phase_reg_kernel<NQ, TAIL, 160, 4>;
    if (block <= 288)
        return phase_reg_kernel<NQ, TAIL, 288, 3>;
    if (block <= 448)
        return phase_reg_kernel<NQ, TAIL, 448, 2>;
    return phase_reg_kernel<NQ, TAIL, 544, 1>;
}

template <int NQ>
RegKernel by_form(int block, int cb, bool dense)
{
    if (block - 32 == cb)
        return by_block<NQ, false>(block, dense);
    if constexpr (NQ == 4 || NQ == 8)
        return by_block<NQ, true>(block, dense);
    return nullptr;
}

}  // namespace

}  // namespace csc
