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
//   P=7, K=25, L=64, T=200,000, 1024 segments   722 -> 521 us
//   P=5, K=18, L=51, T=60,013                   2737 -> 570 us
//   P=1, K=5, L=16, T=2000, 10 segments         734 -> 275 us
//   P=1, K=25, L=200, T=5,000,000               26.8 -> 17.2 ms
// What bounds it now: 2300 cycles per link with one block on an SM (the L2 round
// trip of the coefficients 600-700 of them); with five blocks the L1/shared
// pipe (76% busy).
#pragma once

#include "csc_internal.cuh"
#include "phase_rank.cuh"
#include "phase_reg.cuh"

namespace csc {

namespace {

// Index word of a key (key_index, atoms from bit 17 on): the column's bits.
constexpr int kKeyShift = 17;
__device__ __forceinline__ unsigned key_pos(unsigned slot, unsigned c)
{
    return (slot << 12) | (c << 2);
}

// One launch of a phase.  drain == 0: block b visits segment phase_list[b];
// else the blocks drain the queue (see launch_phase_drain).
// TAIL: several groups of atoms, the last of which may hold fewer than NQ quads.
template <int NQ, bool TAIL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    phase_reg_kernel(PhaseParams pp, int cb, int drain)
{
    constexpr int N = 4 * NQ;
    const float kNan = __int_as_float(0x7fffffff);
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ __align__(16) unsigned long long s_key[2][32];
    constexpr int kAtoms = TAIL ? kRegAtoms : N;  // (without TAIL: one group)
    __shared__ __align__(16) float s_nrm[kAtoms], s_rn[kAtoms];
    // active list: r, z, index word of the key (flags 0), Z' of the last step
    __shared__ __align__(16) float4 s_act[kActive];
    // objective decrease of the visit, in one order whatever lanes hold the nonzeros:
    // update it leaves its term in s_term[it & 63] and the active warp adds every 32 of
    // them to s_dec (double-float).  (A sum per thread depended on the order in which the
    // nonzeros were listed; one FP64 sum by whoever applies the update stands in the
    // chain of updates: 2 to 5% of a solve.  This: under 0.5% of the workloads' solves,
    // 3% of one with K = 128, L = 16, T = 20,000.)
    __shared__ float s_term[64];
    __shared__ float2 s_dec[32];
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
                float v[N];  // (r and Z in one round trip)
                {
                    const float *rp = rbase + jj, *zp = zbase + jj;
#pragma unroll
                    for (int i = 0; i < N; i++, rp += step)
                        v[i] = (int)kbase + i < K ? *rp : 0.f;
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
                rank_column<N>(v, rc, rn, lam, zb, kbase, kKeyShift, pos, khi, klo);
                if (zb)
                    rank_unlisted(zb, rc, zbase + jj, ld, nrm, rn, lam, kbase, kKeyShift, pos, khi,
                                  klo);
                skey[jj] = ((unsigned long long)khi << 32) | klo;
                slst[jj] = zl;
                sunl[jj] = zb;
            }
        __syncthreads();
        int nact = s_nact < kActive ? s_nact : kActive;
        float term = 0.f;  // of this thread's update

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
                        term = delta * (e[x].x - 0.5f * n * delta) + lam * (fabsf(z) - fabsf(u));
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
        if (!is_col) {
            s_term[lane] = s_term[32 + lane] = 0.f;
            s_dec[lane] = make_float2(0.f, 0.f);
            active_step(false, 0u, 0, 0, 0.f);
        }

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
                if ((it & 31) == 0 && it > 0) {
                    const int i = ((it - 1) & 32) + lane;
                    df_add(s_dec[lane].x, s_dec[lane].y, s_term[i]);
                    s_term[i] = 0.f;
                }
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
                            term = delta * (r0 - 0.5f * n * delta) + lam * (fabsf(z) - fabsf(u));
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
                        rank_column<N>(v, rc, rn, lam, zb, kbase, kKeyShift, pos, khi, klo);
                        if (zb)
                            rank_unlisted(zb, rc, zbase + jj, ld, nrm, rn, lam, kbase, kKeyShift, pos,
                                          khi, klo);
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
            if (term != 0.f) {
                s_term[it & 63] = term;
                term = 0.f;
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
        float dec_hi = 0.f, dec_lo = 0.f;
        if (warp == 0) {
            dec_hi = s_dec[lane].x;
            dec_lo = s_dec[lane].y;
            df_add(dec_hi, dec_lo, s_term[((nupd - 1) & 32) + lane]);
#pragma unroll 1
            for (int o = 1; o < 32 && o < nupd; o <<= 1) {  // (most visits: a few terms)
                const float h = __shfl_xor_sync(kFull, dec_hi, o);
                const float l = __shfl_xor_sync(kFull, dec_lo, o);
                df_add_df(dec_hi, dec_lo, h, l);
            }
        }
        if (tid == 0) {
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
                atomicAdd(&pp.dec[slot], (double)dec_hi + (double)dec_lo);
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
// blocks per SM count; else a segment's chain of updates counts (launch_phase_reg has
// the line).  One group of atoms (K <= 32) has a form for every NQ, so no quad is
// padding; with more groups the last one may be short (TAIL).
template <int NQ, bool TAIL>
RegKernel by_block(int block, bool dense)
{
    if (block <= 160)
        return dense ? phase_reg_kernel<NQ, TAIL, 160, 5> : phase_reg_kernel<NQ, TAIL, 160, 4>;
    if (dense && block <= 288)
        return phase_reg_kernel<NQ, TAIL, 288, 3>;
    if (dense && block <= 448)
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
