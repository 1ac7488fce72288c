// FP32 sweeps on the fifth-generation tensor cores: the digit products of sweep_dg.cuh with four digits.
//
// x = 2^(E - 8) sum_{k < 4} d_k 2^(-9 k), |d_0| <= 128, |d_k| <= 256, |x| < 2^(E - 1): 35 bits below the row's
// power of two, so an FP32 entry down to 2^-11 of its row's largest is split exactly.  A term d_k
// 2^(-9 k) is exact in BF16, so products of different orders can share an FP32 accumulator: one takes
// the order 0 (integers below 2^20, exact), the other the orders 3, 2, 1 in turn (below 2^13; what the
// tensor core truncates there lies 2^-24 below it, 2^-9 of an FP32 rounding of the leading sum).
// Orders past 3 are dropped: of the product of the row maxima at most 2^-24 (every digit at its limit, all
// of one sign), about 2^-31 for random digits.  An entry then takes two FP32 roundings where a dot product on
// the FP32 pipes takes 64, and both sweeps run here: S_k^+ came out as exact as with the FP32 pipes
// or up to five times more (against FP64; a split-TF32 update, whose leading sums the tensor core
// truncates, was 1.5 to 19 times less exact than the pipes and stayed out of the pinned sweep).
//
// Kernels of a step over pivot block J (64 wide), on the block upper triangle as in sweep_dg.cuh:
// k_pivot_f32 (the block's inverse in registers), k_panel_d4 (pan = old D^-1 on the FP32 pipes, written
// to M, and the digits of both), k_update_d4, and k_mirror_up at the end.
//
// k_update_d4: one CTA per SM works through an even share of the 128 x 128 blocks, in segments of a
// column of blocks (A = digits of pan for its 128 columns of M, 64 KB, loaded per segment; B = digits of old for
// 128 rows, 64 KB each, two buffers); 2 x 128 accumulator columns, twice, so the 40 MMAs of a
// block (about 68 clocks each) run beside the epilogue of the block before.  Eight epilogue warps keep
// 32 x 32 entries of M in registers and load the next ones meanwhile (sixteen warps had to spill, which waits
// for the loads: 172 us instead of 122).  Per block 128 KB of M and 64 to 128 KB of digits pass through L2;
// copies and M alone took 135 us with a CTA per one or two blocks, the MMAs alone 45.  The entries of J are written by
// k_panel_d4: taken here, lane by lane from pan and D^-1, they doubled the time of the fifth of
// the blocks that meet J or an edge.  Peridynamic factorization workload (16 subdomains, 2700 dofs on average): 122 us
// for a step of all subdomains, 91 us on average against 443 us for split-TF32 over the whole
// matrix; 15 us for the pinned matrices against 146 us on the FP32 pipes.
// Every wait is bounded, as in k_update_dg.
#pragma once

constexpr int D4 = 4;
constexpr int D4_STAGES = 2;
constexpr int D4_SMEM_UPD = (1 + D4_STAGES) * D4 * DG_TBYTES + 1024;
constexpr int D4_ACC = 2 * DG_TILE;                 // accumulator columns of a block
constexpr int D4_XS = DG_TILE + 4;                  // row stride of the staged panel
constexpr int D4_PAN_THREADS = 256;
constexpr int D4_SMEM_PAN = (NB * D4_XS + NB * NB) * 4;

constexpr int D4_EPI = 8;                           // epilogue warps of the update (32 rows of a half block each)
constexpr int D4_THREADS = (D4_EPI + 1) * 32;       // and one for copies and MMAs

struct Digit4Args : SweepArgs<float> {
    unsigned char *pan_d, *old_d;      // digits: per subdomain, per 128-row tile, D4 x 16 KB
    float *pan_s, *old_s;              // per row 2^(E - 8): the product of two scales a sum of digit products
    int *piv_c;                        // per subdomain NB: half the exponent of the pivots (as in k_pivot_dg)
    const int4 *segs;                  // the update's segments: subdomain, column tile, row blocks [q0, q1)
    const int32_t *seg_ptr;            // per CTA: its first segment
};

// Invert the pivot block: 256 threads hold 4 x 4 tiles of the whole symmetric block in registers and
// sweep it by eight pivots at a time: the eight columns go to shared memory (old), every warp inverts
// their 8 x 8 block by itself (two entries per lane, shuffles: 8 dependent steps without a barrier) and
// forms its 8 rows of pan = old D^-1, then all subtract pan old^T.  Bound by the chain of 64
// reciprocals; two barriers per eight pivots.  16 subdomains: 20 us, against 139 us for a shared-memory sweep
// of the whole block and 41 us for k_pivot_dg's layout (a barrier per pivot).  piv_c may be NULL.
constexpr int PIV_THREADS = 256;
constexpr int PIV_W = 8;
__global__ void __launch_bounds__(PIV_THREADS) k_pivot_f32(SweepArgs<float> a, int *piv_c) {
    const int k = blockIdx.x;
    const int pend = a.pend[k];
    if (a.j0 >= pend) return;
    const int b = min(NB, pend - a.j0), ld = a.mld[k];
    const float *M = a.M + a.moff[k];
    __shared__ __align__(16) float old[2][NB][PIV_W], pan[2][NB][PIV_W];
    const int ti = threadIdx.x / 16, tl = threadIdx.x % 16, lane = threadIdx.x % 32, row = threadIdx.x / 4;
    float v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int i = 4 * ti + u, l = 4 * tl + y;
            // upper triangle of M; the identity past the block's width
            v[u][y] = (i < b && l < b) ? M[(int64_t)(a.j0 + min(i, l)) * ld + a.j0 + max(i, l)] : (i == l ? 1.f : 0.f);
        }
    if (piv_c && ti == tl)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int ex = (int)(__float_as_uint(v[u][u]) >> 23);       // with the sign: 0 .. 511
            piv_c[k * NB + 4 * ti + u] = ex > 0 && ex < 0xff ? (ex - 127) >> 1 : 0;
        }
    bool ok = true;
    for (int p0 = 0; p0 < NB; p0 += PIV_W) {
        const int buf = (p0 / PIV_W) & 1, tp = p0 / 4;
        float (*ol)[PIV_W] = old[buf], (*pa)[PIV_W] = pan[buf];
        if ((tl & ~1) == tp)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<float4 *>(&ol[4 * ti + u][4 * (tl & 1)]) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
        __syncthreads();
        // D: lane (row lane / 4, columns 2 (lane mod 4) and the next)
        const int dr = lane / 4, dc = lane % 4;
        float w0 = ol[p0 + dr][2 * dc], w1 = ol[p0 + dr][2 * dc + 1];
#pragma unroll
        for (int p = 0; p < PIV_W; ++p) {
            const float d = __shfl_sync(0xffffffffu, (p & 1) ? w1 : w0, p * 4 + p / 2);
            const float ci = __shfl_sync(0xffffffffu, (p & 1) ? w1 : w0, dr * 4 + p / 2);
            const float r0 = __shfl_sync(0xffffffffu, w0, p * 4 + dc), r1 = __shfl_sync(0xffffffffu, w1, p * 4 + dc);
            if (!(d > 0.f)) ok = false;
            const float inv = 1.f / d, ri = ci * inv;
            const bool c0 = 2 * dc == p, c1 = 2 * dc + 1 == p;
            if (dr == p) {
                w0 = c0 ? -inv : r0 * inv;
                w1 = c1 ? -inv : r1 * inv;
            } else {
                w0 = c0 ? ri : w0 - ri * r0;
                w1 = c1 ? ri : w1 - ri * r1;
            }
        }
        // pan of the warp's rows (thread: row, two columns); rows of the block itself get D^-1
        float o[PIV_W], s0 = 0.f, s1 = 0.f;
        *reinterpret_cast<float4 *>(o) = *reinterpret_cast<const float4 *>(&ol[row][0]);
        *reinterpret_cast<float4 *>(o + 4) = *reinterpret_cast<const float4 *>(&ol[row][4]);
#pragma unroll
        for (int s = 0; s < PIV_W; ++s) {
            s0 -= o[s] * __shfl_sync(0xffffffffu, w0, s * 4 + dc);
            s1 -= o[s] * __shfl_sync(0xffffffffu, w1, s * 4 + dc);
        }
        if (row / PIV_W == p0 / PIV_W) { s0 = -w0; s1 = -w1; }
        *reinterpret_cast<float2 *>(&pa[row][2 * dc]) = make_float2(s0, s1);
        __syncthreads();
        const bool iP = (ti & ~1) == tp, lP = (tl & ~1) == tp;
        if (!iP && !lP) {
#pragma unroll
            for (int h = 0; h < PIV_W; h += 4) {
                float4 pi[4], lo[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    pi[u] = *reinterpret_cast<const float4 *>(&pa[4 * ti + u][h]);
                    lo[u] = *reinterpret_cast<const float4 *>(&ol[4 * tl + u][h]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        v[u][y] -= pi[u].x * lo[y].x;
                        v[u][y] -= pi[u].y * lo[y].y;
                        v[u][y] -= pi[u].z * lo[y].z;
                        v[u][y] -= pi[u].w * lo[y].w;
                    }
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const int i = 4 * ti + u, l = 4 * tl + y;
                    v[u][y] = !lP ? pa[l][i - p0] : (iP ? -pa[i][l - p0] : pa[i][l - p0]);
                }
        }
    }
    if (!ok) atomicMax(a.flag, 1);
    float *D = a.dinv + (int64_t)k * NB * NB;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float o[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) o[y] = (4 * ti + u < b && 4 * tl + y < b) ? -v[u][y] : 0.f;
        *reinterpret_cast<float4 *>(D + (4 * ti + u) * NB + 4 * tl) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// E with |x| < 2^(E - 1), at least -100 (so that every scale below is a normal number)
__device__ __forceinline__ int d4_exp(float x) {
    const int ex = (int)((__float_as_uint(x) >> 23) & 0xff);
    return ex == 0xff ? DG_NAN : max(ex, 25) - 125;
}
__device__ __forceinline__ float d4_pow2(int e) {   // 2^e, e within the normal range
    return __uint_as_float((uint32_t)(e + 127) << 23);
}
__device__ __forceinline__ float d4_scale(int E) { return E >= DG_NAN ? __int_as_float(0x7fc00000) : d4_pow2(E - 8); }

// The panels of 128 rows: pan = old D^-1 (thread: 8 rows x 4 columns, 64 FMAs each in the order of
// the pivots), then the digits of the scaled rows of old and pan (thread: a row, half of its columns),
// written where k_update_d4's copies take them from.  Grid (tiles, K).  One wave of CTAs, bound by
// instructions and its chain of phases: 35 us for 16 x 21 tiles (42 us before, FMAs and copies alone).
__global__ void __launch_bounds__(D4_PAN_THREADS) k_panel_d4(Digit4Args a) {
    const int k = blockIdx.y;
    const int pend = a.pend[k];
    if (a.j0 >= pend) return;
    const int n = a.mdim[k], ld = a.mld[k], tile = blockIdx.x, r0 = tile * DG_TILE;
    if (r0 >= n) return;
    const int b = min(NB, pend - a.j0), j0 = a.j0, jt = j0 / DG_TILE;
    float *M = a.M + a.moff[k];
    extern __shared__ __align__(16) float d4_sm[];
    float *xs = d4_sm, *Ds = d4_sm + NB * D4_XS;      // xs[column][row], D^-1
    __shared__ int se[2][DG_TILE], spc[NB];
    const int t = threadIdx.x, r = t % DG_TILE, h = t / DG_TILE;
    for (int q = t; q < NB * NB; q += D4_PAN_THREADS) Ds[q] = a.dinv[(int64_t)k * NB * NB + q];
    if (t < NB) spc[t] = a.piv_c[k * NB + t];
    // rows of the tiles up to the pivot's hold M_iJ, those below are read from the transposed block
    // (the pivot's own diagonal tile is whole)
    if (tile <= jt) {
#pragma unroll 8
        for (int q = t; q < NB * DG_TILE; q += D4_PAN_THREADS) {
            const int c = q % NB, i = q / NB;
            xs[c * D4_XS + i] = r0 + i < n && c < b ? M[(int64_t)(r0 + i) * ld + j0 + c] : 0.f;
        }
    } else {
#pragma unroll 8
        for (int q = t; q < NB * DG_TILE; q += D4_PAN_THREADS) {
            const int c = q / DG_TILE, i = q % DG_TILE;
            xs[c * D4_XS + i] = r0 + i < n && c < b ? M[(int64_t)(j0 + c) * ld + r0 + i] : 0.f;
        }
    }
    __syncthreads();
    const int64_t row0 = a.scr_off[k] + r0, tile_off = row0 / DG_TILE * D4 * DG_TBYTES;
    // digits of the rows in xs, columns scaled by 2^(sg c_s); every thread calls it
    auto split = [&](unsigned char *dst, float *scale, int sg) {
        float x[NB / 2];
        int E = -100;
#pragma unroll
        for (int s = 0; s < NB / 2; ++s) {
            const int c = h * (NB / 2) + s;
            x[s] = xs[c * D4_XS + r] * d4_pow2(sg * spc[c]);
            E = max(E, d4_exp(x[s]));
        }
        se[h][r] = E;
        __syncthreads();
        E = max(se[0][r], se[1][r]);
        if (h == 0) scale[row0 + r] = d4_scale(E);
        const float f = E >= DG_NAN ? 0.f : d4_pow2(8 - E);
#pragma unroll
        for (int s = 0; s < NB / 2; ++s) x[s] *= f;
        // digit q: x rounded to a multiple of 2^(-9 q) by adding and subtracting 1.5 2^(23 - 9 q); exact
        // in BF16, the upper half of its FP32 word
#pragma unroll
        for (int q = 0; q < D4; ++q) {
            const float mg = 1.5f * d4_pow2(23 - 9 * q);
#pragma unroll
            for (int s = 0; s < NB / 2; s += 8) {
                uint32_t o[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float &x0 = x[s + 2 * e], &x1 = x[s + 2 * e + 1];
                    const float d0 = __fsub_rn(__fadd_rn(x0, mg), mg), d1 = __fsub_rn(__fadd_rn(x1, mg), mg);
                    x0 = __fsub_rn(x0, d0);
                    x1 = __fsub_rn(x1, d1);
                    o[e] = __byte_perm(__float_as_uint(d0), __float_as_uint(d1), 0x7632);
                }
                *reinterpret_cast<uint4 *>(dst + q * DG_TBYTES + dg_off(r, h * (NB / 2) + s)) =
                    make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    };
    split(a.old_d + tile_off, a.old_s, -1);
    // pan
    const int tx = t % 16, ty = t / 16;
    float2 ap[4][4];                    // pairs of rows: packed FMAs, each half rounded as the scalar one
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) ap[u][v] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int s = 0; s < b; ++s) {
        const float4 d = *reinterpret_cast<const float4 *>(Ds + s * NB + 4 * tx);
        const float4 p = *reinterpret_cast<const float4 *>(xs + s * D4_XS + 8 * ty);
        const float4 w = *reinterpret_cast<const float4 *>(xs + s * D4_XS + 8 * ty + 4);
        const float2 xr[4] = {make_float2(p.x, p.y), make_float2(p.z, p.w), make_float2(w.x, w.y), make_float2(w.z, w.w)};
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) ap[u][v] = __ffma2_rn(xr[u], make_float2(dv[v], dv[v]), ap[u][v]);
    }
    float acc[8][4];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = (u & 1) ? ap[u / 2][v].y : ap[u / 2][v].x;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) xs[(4 * tx + v) * D4_XS + 8 * ty + u] = acc[u][v];
    __syncthreads();
    // M_iJ = pan (-D^-1 for the rows of J), where M_iJ was read; in the pivot's diagonal tile, which is
    // whole, also the transposed entries of the other rows.  k_update_d4 leaves J alone
    if (tile <= jt) {
#pragma unroll 8
        for (int q = t; q < NB * DG_TILE; q += D4_PAN_THREADS) {
            const int c = q % NB, i = q / NB, ij = r0 + i - j0;
            if (r0 + i < n && c < b) M[(int64_t)(r0 + i) * ld + j0 + c] = ij >= 0 && ij < b ? -Ds[ij * NB + c] : xs[c * D4_XS + i];
        }
    }
    if (tile >= jt) {
#pragma unroll 8
        for (int q = t; q < NB * DG_TILE; q += D4_PAN_THREADS) {
            const int c = q / DG_TILE, i = q % DG_TILE, ij = r0 + i - j0;
            if (r0 + i < n && c < b && (ij < 0 || ij >= b)) M[(int64_t)(j0 + c) * ld + r0 + i] = xs[c * D4_XS + i];
        }
    }
    split(a.pan_d + tile_off, a.pan_s, 1);
}

// the digit products of a 128 x 128 block: order 0 in the first 128 accumulator columns, orders 3, 2, 1 in
// the second.  BF16 operands (format 1 at bits 7-9 and 10-12 of the descriptor)
__device__ __forceinline__ void d4_products(uint32_t tmem, uint32_t a, uint32_t b) {
    constexpr uint32_t IDESC = dg_idesc(DG_TILE, DG_TILE) | (1u << 7) | (1u << 10);
    const uint64_t da = tc_desc(a), db = tc_desc(b);
#pragma unroll
    for (int d = D4 - 1; d >= 0; --d)
#pragma unroll
        for (int i = 0; i <= d; ++i)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)          // K = 16: 32 bytes along the row
                dg_mma(tmem + (d > 0 ? DG_TILE : 0), da + (uint64_t)((i * DG_TBYTES + 32 * kk) >> 4),
                       db + (uint64_t)(((d - i) * DG_TBYTES + 32 * kk) >> 4), IDESC,
                       ((d > 0 && d < D4 - 1) || i > 0 || kk > 0) ? 1 : 0);
}

// grid: at most one CTA per SM, each with its segments of the columns' blocks (of the subdomains that have
// pivots left)
__global__ void __launch_bounds__(D4_THREADS, 1) k_update_d4(Digit4Args a) {
    const int sg0 = a.seg_ptr[blockIdx.x], sg1 = a.seg_ptr[blockIdx.x + 1];
    const int j0 = a.j0;
    extern __shared__ __align__(1024) unsigned char dg_raw[];
    unsigned char *sa = dg_raw + ((1024u - (tc_s32(dg_raw) & 1023u)) & 1023u), *sb = sa + D4 * DG_TBYTES;
    __shared__ uint64_t full_a, full_b[D4_STAGES], empty_b[D4_STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        dg_bar_init(&full_a, 1);
        for (int s = 0; s < D4_STAGES; ++s) {
            dg_bar_init(&full_b[s], 1);
            dg_bar_init(&empty_b[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            dg_bar_init(&acc_full[s], 1);
            dg_bar_init(&acc_empty[s], D4_EPI * 32);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == D4_EPI) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_s32(&tmem_base)),
                     "r"(2 * D4_ACC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    if (warp == D4_EPI) {
        // ------------------------------------------------------------ copies and MMAs, one thread
        if (lane == 0) {
            // B of the next block of the CTA, whatever its segment
            int loaded = 0, lsg = sg0, a_loads = 0;
            int4 lseg = a.segs[sg0];
            auto load_b = [&]() {
                if (lsg >= sg1) return;
                const int s = loaded++ % D4_STAGES;
                dg_bar_expect(&full_b[s], D4 * DG_TBYTES);
                dg_g2s(sb + s * D4 * DG_TBYTES, a.old_d + (a.scr_off[lseg.x] / DG_TILE + lseg.z) * D4 * DG_TBYTES,
                       D4 * DG_TBYTES, &full_b[s]);
                if (++lseg.z == lseg.w && ++lsg < sg1) lseg = a.segs[lsg];
            };
            bool ok = true;
            int it = 0;
            for (int sg = sg0; sg < sg1 && ok; ++sg) {
                const int4 seg = a.segs[sg];
                // A of the segment's column, once the MMAs that read the one before are done
                if (it > 0) ok = tc_wait(&empty_b[(it - 1) % D4_STAGES], ((it - 1) / D4_STAGES) & 1, TC_WAIT_TRIES);
                if (!ok) break;
                dg_bar_expect(&full_a, D4 * DG_TBYTES);
                dg_g2s(sa, a.pan_d + (a.scr_off[seg.x] / DG_TILE + seg.y) * D4 * DG_TBYTES, D4 * DG_TBYTES, &full_a);
                ++a_loads;
                if (it == 0)
                    for (int s = 0; s < D4_STAGES; ++s) load_b();
                ok = tc_wait(&full_a, (a_loads - 1) & 1, TC_WAIT_TRIES);
                for (int q = seg.z; q < seg.w && ok; ++q) {
                    const int s = it % D4_STAGES, ab = it & 1;
                    // the accumulators were last drained for block it - 2
                    ok = !abort_flag && tc_wait(&full_b[s], (it / D4_STAGES) & 1, TC_WAIT_TRIES) &&
                         (it < 2 || tc_wait(&acc_empty[ab], ((it - 2) >> 1) & 1, TC_WAIT_TRIES));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    d4_products(tmem + (uint32_t)(ab * D4_ACC), tc_s32(sa), tc_s32(sb + s * D4 * DG_TBYTES));
                    dg_commit(&acc_full[ab]);
                    dg_commit(&empty_b[s]);
                    ++it;
                    // refill the buffer the block before used (its MMAs are done once empty_b fires)
                    if (it >= 2 && lsg < sg1) {
                        ok = tc_wait(&empty_b[(it - 2) % D4_STAGES], ((it - 2) / D4_STAGES) & 1, TC_WAIT_TRIES);
                        if (ok) load_b();
                    }
                }
            }
            if (!ok) {
                atomicExch(a.flag + 2, 1);
                abort_flag = 1;
            }
            // what was copied has landed and what was issued is done before the CTA goes
            if (a_loads > 0) tc_wait(&full_a, (a_loads - 1) & 1, TC_WAIT_TRIES);
            for (int x = max(0, loaded - D4_STAGES); x < loaded; ++x)
                tc_wait(&full_b[x % D4_STAGES], (x / D4_STAGES) & 1, TC_WAIT_TRIES);
            for (int x = max(0, it - 2); x < it; ++x)
                tc_wait(&empty_b[x % D4_STAGES], (x / D4_STAGES) & 1, TC_WAIT_TRIES);
        }
    } else {
        // ------------------------------------------------------------ epilogue: column i of M per lane
        const int qd = warp & 3, hf = warp >> 2;      // lane quarter; 32 of the 64 rows of a half block
        int it = 0;
        bool go = true;
        for (int sg = sg0; sg < sg1 && go; ++sg) {
        const int4 seg = a.segs[sg];
        const int k = seg.x, c0 = seg.y * DG_TILE, n = a.mdim[k], ld = a.mld[k], j1 = j0 + min(NB, a.pend[k] - j0);
        const int64_t row0 = a.scr_off[k];
        float *M = a.M + a.moff[k];
        const int i = c0 + 32 * qd + lane;
        const bool in = i < n, iJ = i >= j0 && i < j1;
        const float sc = in ? a.pan_s[row0 + i] : 0.f;
        // a half block of the warp, 32 rows x 32 columns of M, and the rows' scales (a lane each); loaded
        // one half ahead of their use
        struct Half { float m[32], s; };
        Half ha, hb;
        auto load_half = [&](int h, Half &v) {
            const int l0 = h * DG_LB + 32 * hf;
            v.s = a.old_s[row0 + l0 + lane];
            const float *Mp = M + (int64_t)l0 * ld + i;
            if (l0 + 32 <= n && c0 + DG_TILE <= n) {
#pragma unroll
                for (int c = 0; c < 32; ++c) v.m[c] = Mp[(int64_t)c * ld];
            } else {
#pragma unroll
                for (int c = 0; c < 32; ++c) v.m[c] = in && l0 + c < n ? Mp[(int64_t)c * ld] : 0.f;
            }
        };
        // waits for the accumulators (half 0), subtracts, stores; false: given up
        auto half_block = [&](int h, Half &v) {
            const int ab = it & 1, l0 = h * DG_LB + 32 * hf;
            if (!(h & 1)) {
                const bool ok = !abort_flag && tc_wait(&acc_full[ab], (it >> 1) & 1, TC_WAIT_TRIES);
                if (__any_sync(0xffffffffu, !ok)) {
                    if (lane == 0) {
                        atomicExch(a.flag + 2, 1);
                        abort_flag = 1;
                    }
                    return false;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
            const uint32_t ta = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(ab * D4_ACC + (h & 1) * DG_LB + 32 * hf);
#pragma unroll
            for (int cc = 0; cc < 32; cc += 8) {
                __syncwarp();                       // the half block before branched at its stores; the loads are .aligned
                uint32_t a0[8], a1[8];
                dg_ld8(ta + (uint32_t)cc, a0);
                dg_ld8(ta + (uint32_t)(DG_TILE + cc), a1);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (cc == 24 && (h & 1)) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    dg_bar_arrive(&acc_empty[ab]);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float x = __fadd_rn(__uint_as_float(a0[c]), __uint_as_float(a1[c]));
                    v.m[cc + c] = __fmaf_rn(-(x * sc), __shfl_sync(0xffffffffu, v.s, cc + c), v.m[cc + c]);
                }
            }
            float *Mp = M + (int64_t)l0 * ld + i;
            // plain when the pivot block and the edges are elsewhere
            if (c0 + DG_TILE <= n && l0 + 32 <= n && (j1 <= c0 || j0 >= c0 + DG_TILE) && (j1 <= l0 || j0 >= l0 + 32)) {
#pragma unroll
                for (int c = 0; c < 32; ++c) Mp[(int64_t)c * ld] = v.m[c];
            } else if (in && !iJ) {                     // J holds its new values already
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int l = l0 + c;
                    if (l < n && (l < j0 || l >= j1)) Mp[(int64_t)c * ld] = v.m[c];
                }
            }
            return true;
        };
        load_half(2 * seg.z, ha);
        for (int q = seg.z; q < seg.w; ++q, ++it) {
            load_half(2 * q + 1, hb);
            go = half_block(2 * q, ha);
            if (!go) break;
            if (q + 1 < seg.w) load_half(2 * q + 2, ha);
            half_block(2 * q + 1, hb);
        }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == D4_EPI) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * D4_ACC) : "memory");
    }
}
