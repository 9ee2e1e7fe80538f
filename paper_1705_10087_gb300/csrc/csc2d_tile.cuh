// The 2-D tile visit with thread-private positions (included by csc2d.cu): the
// counterpart of the 1-D form in phase_reg_impl.cuh.
//
// Thread (a, b) of the position threads owns the positions of the tile and of
// the h-1 rows and w-1 columns around it (its halo) whose row is a (mod 2h-1)
// and whose column is b (mod 2w-1), counted from the halo's corner: a window's
// (2h-1)(2w-1) positions go to distinct threads.  The r of tile and halo are
// staged in shared memory, a position's atoms one after the other; the halo (an
// idle neighbour's positions, which no other block of the launch touches) comes
// in the background and is written back once where it changed.  Atomic additions
// to the neighbours, 44% of an update's window for a 14 x 14 tile with 15 x 15
// windows, were most of an update's time.  Coordinates with z != 0 belong to the
// active warp, one lane each.  Order of updates, ties and roundings are those of
// tile_kernel.
//
// What bounds it is the latency of an update (argmax, barrier, coefficients,
// ranking), about 2.1 us, and 7 us per launch for the flags, the tile and its halo.
// 512 x 512 image, 8 atoms of 8 x 8, 36 x 36 tiles, 96 launches: 2483 us with
// tile_kernel, 1472 us with this form.
#pragma once

#include "phase_rank.cuh"

namespace {

using namespace csc;

constexpr int kPosWarps = 16;  // position warps of a block at most (and the active warp)
constexpr int kTileRegSmem = kMaxSmem - 4096;  // dynamic shared memory at most (static: 3 KB)

// Shared memory (bytes): ext positions of NQ | 1 quads (tile and halo), and per tile
// position a key and the bits of its listed and unlisted nonzeros.
__host__ __device__ constexpr size_t tile_reg_smem(int nq, int64_t ext, int64_t own)
{
    return (size_t)ext * 16 * (nq | 1) + (size_t)own * 16;
}

template <int NQ, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) tile_reg_kernel(TileParams tp)
{
    constexpr int N = 4 * NQ;
    constexpr int kStride = (NQ | 1) * 2;  // pairs of a position
    const float kNan = __int_as_float(0x7fffffff);
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ __align__(16) unsigned long long s_key[2][32];
    __shared__ __align__(16) float nrm[N], rn[N];
    // active list: r, z, index word of the key (flags 0), Z' of the last step
    __shared__ __align__(16) float4 s_act[kActive];
    __shared__ double s_dec[kPosWarps + 1];
    __shared__ int s_nact;

    const int tile = tp.list[blockIdx.x];
    if (!tp.dirty[tile])
        return;  // uniform: every thread reads the same flag
    const int m = tile / tp.Mc, n = tile % tp.Mc;
    const Dims d = tp.d;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const bool is_pos = tid < (int)blockDim.x - 32;  // the last warp has the active list
    const int K = d.K, KQ = tp.KQ, h1 = d.h - 1, w1 = d.w - 1;
    const int H2 = 2 * d.h - 1, W2 = 2 * d.w - 1, A = H2 * W2;
    const int64_t i_lo = tp.row_s[m], i_hi = tp.row_s[m + 1];
    const int64_t j_lo = tp.col_s[n], j_hi = tp.col_s[n + 1];
    const int th = (int)(i_hi - i_lo), tw = (int)(j_hi - j_lo);
    const int EH = th + 2 * h1, EW = tw + 2 * w1;
    const int64_t Wz = d.Wz, HWz = d.Hz * d.Wz;
    // valid rows and columns of the tile with its halo
    const int row_lo = i_lo < h1 ? (int)(h1 - i_lo) : 0, col_lo = j_lo < w1 ? (int)(w1 - j_lo) : 0;
    const int row_hi = d.Hz - i_lo + h1 < EH ? (int)(d.Hz - i_lo + h1) : EH;
    const int col_hi = Wz - j_lo + w1 < EW ? (int)(Wz - j_lo + w1) : EW;
    const int a = tid / W2, b = tid - a * W2;  // (a >= H2: no position)
    const float lam = tp.lam, tol = tp.tol;
    // element (k, row, col) of the halo's frame at + k HWz + row Wz + col
    const int64_t corner = (i_lo - h1) * Wz + (j_lo - w1);
    float *const rg = tp.r + corner;
    float *const zg = tp.Z + corner;
    unsigned long long *const rs = reinterpret_cast<unsigned long long *>(sm);
    unsigned long long *const keys = rs + (size_t)tp.max_ext * kStride;
    unsigned *const slst = reinterpret_cast<unsigned *>(keys + tp.max_pos);
    unsigned *const sunl = slst + tp.max_pos;
    // index word: k << kshift | row << (2 + jbits) | col << 2 | listed | sign, rows
    // and columns of the tile: ties go to the lowest (k Hz + i) Wz + j
    const int jbits = tw > 1 ? 32 - __clz(tw - 1) : 0;
    const int ibits = th > 1 ? 32 - __clz(th - 1) : 0;
    const int kshift = 2 + ibits + jbits;
    const unsigned jmask = (1u << jbits) - 1u, imask = (1u << ibits) - 1u;
    // one position of the tile per thread at most: its key stays in khi, klo
    const bool single = th <= H2 && tw <= W2;
    const int nc = (EW + W2 - 1) / W2;  // positions of a thread along a row

    for (int k = tid; k < N; k += blockDim.x) {
        // (rn = 0 beyond the last atom: no excess there)
        nrm[k] = k < K ? tp.norms[k] : 1.f;
        rn[k] = k < K ? __frcp_rn(tp.norms[k]) : 0.f;
    }
    if (tid < 64)
        s_key[tid >> 5][tid & 31] = 0ull;
    if (tid == 0)
        s_nact = 0;
    __syncthreads();

    unsigned khi = 0, klo = 0;  // single: the position's key; active lane: its best
    unsigned changed = 0;       // the thread's positions whose r changed
    // f(slot bit, row, col) over the thread's positions in the frame
    auto for_positions = [&](auto &&f) {
        if (a >= H2)
            return;
#pragma unroll 1
        for (int row = a, sr = 0; row < EH; row += H2, sr++)
#pragma unroll 1
            for (int col = b, sc = 0; col < EW; col += W2, sc++)
                if (row >= row_lo && row < row_hi && col >= col_lo && col < col_hi)
                    f(sr * nc + sc, row, col);
    };
    auto inside = [&](int row, int col) {
        return row >= h1 && row < h1 + th && col >= w1 && col < w1 + tw;
    };
    if (is_pos) {
        for_positions([&](int, int row, int col) {
            if (!inside(row, col))
                halo_load<N>(rs + (row * EW + col) * kStride, rg + row * Wz + col, HWz, K);
        });
        for_positions([&](int, int row, int col) {
            if (!inside(row, col))
                return;
            const int ii = row - h1, jj = col - w1, o = ii * tw + jj;
            const unsigned pos = ((unsigned)ii << (2 + jbits)) | ((unsigned)jj << 2);
            const int64_t at = row * Wz + col;
            const int64_t step = opaque(HWz);
            unsigned zb = 0, zl = 0;
            float v[N];  // (r and Z in one round trip)
            {
                const float *rp = rg + at, *zp = zg + at;
#pragma unroll
                for (int i = 0; i < N; i++, rp += step)
                    v[i] = i < K ? *rp : 0.f;
#pragma unroll
                for (int i = 0; i < N; i++, zp += step)
                    zb |= (i < K && *zp != 0.f ? 1u : 0u) << i;
            }
#pragma unroll 1
            for (unsigned rest = zb; rest; rest &= rest - 1) {
                const int i = __ffs((int)rest) - 1, e = atomicAdd(&s_nact, 1);
                if (e < kActive) {
                    s_act[e] = make_float4(rg[at + i * step], zg[at + i * step],
                                           __uint_as_float(((unsigned)i << kshift) | pos), 0.f);
                    zl |= 1u << i;
                }
            }
            zb &= ~zl;
#pragma unroll
            for (int i = 0; i < N; i++)
                if (zl >> i & 1u)
                    v[i] = kNan;
            unsigned long long *const col2 = rs + (row * EW + col) * kStride;
#pragma unroll
            for (int q = 0; q < NQ; q++) {
                const ulonglong2 n4 = *reinterpret_cast<const ulonglong2 *>(rn + 4 * q);
                const ulonglong2 x = make_ulonglong2(pack2(v[4 * q], v[4 * q + 1]),
                                                     pack2(v[4 * q + 2], v[4 * q + 3]));
                *reinterpret_cast<ulonglong2 *>(col2 + 2 * q) = x;
                excess2(x.x, n4.x, lam, v[4 * q], v[4 * q + 1]);
                excess2(x.y, n4.y, lam, v[4 * q + 2], v[4 * q + 3]);
            }
            if (zb) {
#pragma unroll
                for (int i = 0; i < N; i++)
                    if (zb >> i & 1u)
                        v[i] = -1.f;
            }
            const float *const rc = reinterpret_cast<const float *>(col2);
            rank_column<N>(v, rc, rn, lam, zb, 0u, kshift, pos, khi, klo);
            if (zb)
                rank_unlisted(zb, rc, zg + at, HWz, nrm, rn, lam, 0u, kshift, pos, khi, klo);
            keys[o] = ((unsigned long long)khi << 32) | klo;
            slst[o] = zl;
            sunl[o] = zb;
        });
    }
    __syncthreads();
    int nact = s_nact < kActive ? s_nact : kActive;
    float decrease = 0.f;

    // the lane's listed coordinates after the update (k0, tile position (ii0, jj0),
    // dZ) of key index word win (none of them with upd = false); leaves the lane's
    // best key in khi, klo
    auto active_step = [&](bool upd, unsigned win, int k0, int ii0, int jj0, float delta) {
        khi = klo = 0u;
#pragma unroll 1
        for (int e0 = lane; e0 < nact; e0 += 32) {
            float4 e = s_act[e0];
            const unsigned id = __float_as_uint(e.z), k = id >> kshift;
            const int ii = (int)(id >> (2 + jbits) & imask), jj = (int)(id >> 2 & jmask);
            const float nk = nrm[k];
            if (upd) {
                const int di = ii - ii0 + h1, dj = jj - jj0 + w1;
                float cv = 0.f;
                if (di >= 0 && di < H2 && dj >= 0 && dj < W2)
                    cv = __ldg(tp.Ct +
                               ((((int64_t)k0 * KQ + (k >> 2)) * A + di * W2 + dj) << 2) + (k & 3));
                if ((id | 2u) == (win & ~1u)) {
                    // Prop. A.1 from r before this update touches it:
                    // dZ (r - n dZ / 2) + lam (|z| - |u|)
                    const float u = e.w, z = u - delta;
                    decrease += delta * (e.x - 0.5f * nk * delta) + lam * (fabsf(z) - fabsf(u));
                    e.y = u;
                    zg[k * HWz + (ii + h1) * Wz + jj + w1] = u;
                }
                e.x = fmaf(-cv, delta, e.x);
            }
            float zn, dz;
            coord_step(e.x, e.y, nk, rn[k], lam, &zn, &dz);
            e.w = zn;
            s_act[e0] = e;
            const unsigned h = __float_as_uint(fabsf(dz));
            const unsigned l = ~(id | 2u | (dz < 0.f ? 1u : 0u));
            if (fabsf(dz) > 0.f && (h > khi || (h == khi && l > klo))) {
                khi = h;
                klo = l;
            }
        }
    };
    if (!is_pos)
        active_step(false, 0u, 0, 0, 0, 0.f);

    const char *const Ctb = reinterpret_cast<const char *>(tp.Ct);
    int nupd = 0;
    int imin = th, imax = -1, jmin = tw, jmax = -1;
    bool capped = false;
#pragma unroll 1
    for (int it = 0;; it++) {
        // ---- block argmax of the keys ------------------------------------
        unsigned mh = khi, ml = klo;
        if (is_pos && !single) {
            unsigned long long my = 0ull;
            for_positions([&](int, int row, int col) {
                if (inside(row, col)) {
                    const unsigned long long x = keys[(row - h1) * tw + col - w1];
                    my = x > my ? x : my;
                }
            });
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
        // (kept in ordinary registers: the uniform unit's latency is longer)
        best = (unsigned long long)opaque((int64_t)best);
        const float adz = __uint_as_float((unsigned)(best >> 32));
        if (!(adz >= tol))
            break;
        if (nupd >= tp.u) {
            capped = true;
            break;
        }
        // the winner and dZ = +-|dZ| from its key
        const unsigned flat = ~(unsigned)best;
        const int k0 = (int)(flat >> kshift);
        const int ii0 = (int)(flat >> (2 + jbits) & imask), jj0 = (int)(flat >> 2 & jmask);
        const bool listed = flat & 2u;
        const float delta = (flat & 1u) ? -adz : adz;
        const unsigned long long ndelta = pack2(-delta, -delta);
        // a winner from a position thread is listed from the next update on
        const int slot_new = nact;
        const bool to_list = !listed && nact < kActive;

        if (!is_pos) {
            active_step(true, flat, k0, ii0, jj0, delta);
        } else if (a < H2) {
            // the window covers rows ii0 .. ii0 + 2h-2 of the frame: this
            // thread's row is the one that is a (mod 2h-1), its column likewise
            int oi = a - (th <= H2 ? ii0 : ii0 % H2), oj = b - (tw <= W2 ? jj0 : jj0 % W2);
            oi += oi < 0 ? H2 : 0;
            oj += oj < 0 ? W2 : 0;
            const int row = ii0 + oi, col = jj0 + oj;
            if (row >= row_lo && row < row_hi && col >= col_lo && col < col_hi) {
                // coefficients of (k0, lag): float4 group q at ((k0 KQ + q) A + lag)
                unsigned long long cv[2 * NQ];
                {
                    unsigned o = (unsigned)(k0 * KQ * A + oi * W2 + oj) * 16u;
#pragma unroll
                    for (int q = 0; q < NQ; q++, o += (unsigned)A * 16u) {
                        const ulonglong2 y = __ldg(reinterpret_cast<const ulonglong2 *>(Ctb + o));
                        cv[2 * q] = y.x;
                        cv[2 * q + 1] = y.y;
                    }
                }
                unsigned long long *const col2 = rs + (row * EW + col) * kStride;
                const int sr = row < H2 ? 0 : row < 2 * H2 ? 1 : row / H2;
                const int sc = col < W2 ? 0 : col < 2 * W2 ? 1 : col / W2;
                changed |= 1u << (sr * nc + sc);
                if (inside(row, col)) {
                    const int ii = row - h1, jj = col - w1;
                    const int64_t at = row * Wz + col;
                    float *const rc = reinterpret_cast<float *>(col2);
                    // (none is unlisted while the list has room)
                    unsigned zb = nact < kActive ? 0u : sunl[ii * tw + jj];
                    const unsigned pos = ((unsigned)ii << (2 + jbits)) | ((unsigned)jj << 2);
                    if (ii == ii0 && jj == jj0 && !listed) {
                        const unsigned bit = 1u << k0;
                        const float nk = nrm[k0], r0 = rc[k0];
                        float *const zp = zg + k0 * HWz + at;
                        float u = delta, z = 0.f;
                        if (to_list) {
                            s_act[slot_new] =
                                make_float4(fmaf(-nk, delta, r0), u,
                                            __uint_as_float(((unsigned)k0 << kshift) | pos), u);
                            slst[ii * tw + jj] |= bit;
                            rc[k0] = kNan;
                        } else {
                            // the list is full: Z' as the key's step found it
                            float dz;
                            coord_step(r0, zb & bit ? *zp : 0.f, nk, rn[k0], lam, &u, &dz);
                            z = u - delta;
                            zb = u != 0.f ? (zb | bit) : (zb & ~bit);
                            sunl[ii * tw + jj] = zb;
                        }
                        // Prop. A.1 from r before this update touches it:
                        // dZ (r - n dZ / 2) + lam (|z| - |u|)
                        decrease += delta * (r0 - 0.5f * nk * delta) + lam * (fabsf(z) - fabsf(u));
                        *zp = u;
                    }
                    float v[N];
#pragma unroll
                    for (int q = 0; q < NQ; q++) {
                        const ulonglong2 n4 = *reinterpret_cast<const ulonglong2 *>(rn + 4 * q);
                        ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(col2 + 2 * q);
                        x.x = fma2(cv[2 * q], ndelta, x.x);
                        x.y = fma2(cv[2 * q + 1], ndelta, x.y);
                        *reinterpret_cast<ulonglong2 *>(col2 + 2 * q) = x;
                        excess2(x.x, n4.x, lam, v[4 * q], v[4 * q + 1]);
                        excess2(x.y, n4.y, lam, v[4 * q + 2], v[4 * q + 3]);
                    }
                    if (zb) {
#pragma unroll
                        for (int i = 0; i < N; i++)
                            if (zb >> i & 1u)
                                v[i] = -1.f;
                    }
                    rank_column<N>(v, rc, rn, lam, zb, 0u, kshift, pos, khi, klo);
                    if (zb)
                        rank_unlisted(zb, rc, zg + at, HWz, nrm, rn, lam, 0u, kshift, pos, khi,
                                      klo);
                    if (!single)
                        keys[ii * tw + jj] = ((unsigned long long)khi << 32) | klo;
                } else {
                    // an idle neighbour's position: product and sum rounded one
                    // after the other (as by an atomic addition)
                    halo_wait();
#pragma unroll
                    for (int q = 0; q < NQ; q++) {
                        ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(col2 + 2 * q);
                        x.x = add2(x.x, mul2(cv[2 * q], ndelta));
                        x.y = add2(x.y, mul2(cv[2 * q + 1], ndelta));
                        *reinterpret_cast<ulonglong2 *>(col2 + 2 * q) = x;
                    }
                }
            }
        }
        nact += to_list ? 1 : 0;
        nupd++;
        imin = ii0 < imin ? ii0 : imin;
        imax = ii0 > imax ? ii0 : imax;
        jmin = jj0 < jmin ? jj0 : jmin;
        jmax = jj0 > jmax ? jj0 : jmax;
    }

    // ---- write back, spill bookkeeping (Z was written as it was applied) ---
    halo_wait();
    if (is_pos) {
        for_positions([&](int s, int row, int col) {
            if (!(changed >> s & 1u))
                return;
            const bool own = inside(row, col);
            const unsigned skip = own ? slst[(row - h1) * tw + col - w1] : 0u;
            const float *const rc =
                reinterpret_cast<const float *>(rs + (row * EW + col) * kStride);
            float *dst = rg + row * Wz + col;
            const int64_t step = opaque(HWz);
#pragma unroll
            for (int i = 0; i < N; i++, dst += step)
                if (i < K && !(skip >> i & 1u))
                    *dst = rc[i];
        });
    } else if (nupd > 0) {
        for (int e0 = lane; e0 < nact; e0 += 32) {
            const float4 e = s_act[e0];
            const unsigned id = __float_as_uint(e.z);
            const int ii = (int)(id >> (2 + jbits) & imask), jj = (int)(id >> 2 & jmask);
            rg[(int64_t)(id >> kshift) * HWz + (ii + h1) * Wz + jj + w1] = e.x;
        }
    }
    for (int off = 16; off > 0; off >>= 1)
        decrease += __shfl_xor_sync(0xffffffffu, decrease, off);
    if (lane == 0)
        s_dec[warp] = (double)decrease;
    __syncthreads();
    if (tid == 0) {
        double dsum = 0.0;
        for (int q = 0; q < nwarps; q++)
            dsum += s_dec[q];
        tile_done(tp, tile, m, n, nupd, capped, dsum, i_lo + imin, i_lo + imax, j_lo + jmin,
                  j_lo + jmax);
    }
}

using TileKernel = void (*)(TileParams);

// registers: 65536 / (threads x blocks per SM) at most.  Blocks of 161 to 288 threads
// (windows of 129 to 256 positions): three per SM, so that 456 tiles run at once, at 72
// registers and with spills beyond 8 atoms.  With two per SM (96 registers) many tiles
// are slower, few are faster, calls with 8 x 8 atoms: 1024 x 1024 with K = 8 and K = 2
// 4.18 and 1.21 ms instead of 4.02 and 1.14; 512 x 512, K = 8 2.52 instead of 2.58;
// 256 x 256 with K = 16 7.9 instead of 10.1.
template <int NQ>
TileKernel tile_reg_block(int block)
{
    if (block <= 160)
        return tile_reg_kernel<NQ, 160, 4>;
    if (block <= 288)
        return tile_reg_kernel<NQ, 288, 3>;
    return tile_reg_kernel<NQ, 544, 1>;
}

// The kernel for K atoms (at most 32) and blocks of `block` threads.
TileKernel tile_reg_fn(int K, int block)
{
    switch ((K + 3) / 4) {
    case 1:
        return tile_reg_block<1>(block);
    case 2:
        return tile_reg_block<2>(block);
    case 3:
        return tile_reg_block<3>(block);
    case 4:
        return tile_reg_block<4>(block);
    case 5:
        return tile_reg_block<5>(block);
    case 6:
        return tile_reg_block<6>(block);
    case 7:
        return tile_reg_block<7>(block);
    }
    return tile_reg_block<8>(block);
}

}  // namespace
