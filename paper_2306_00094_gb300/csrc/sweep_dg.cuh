// FP64 sweeps on the fifth-generation tensor cores: products of digit slices, accumulated exactly.
//
// FP64 runs at 1/64 of the FP32 rate on this GPU (two FMAs per SM and clock), and a sweep is 2 n^2 64
// FP64 operations per pivot block: on the pipes it stood at the FP64 peak (6 x 6 table row, 36
// subdomains of about 2100 dofs: 15.3 ms per step, 421 ms in all).  Here every row of a panel is
// written as a power of two times integers of 9 bits (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication by using fast routines of
// matrix multiplication and its applications", 2012):
//   x = 2^(E - 8) sum_{k < DG} d_k 2^(-9 k),  |d_k| <= 256, |d_0| <= 128, |x| < 2^(E - 1),
// DG = 7 digits, 61 bits below the row's power of two.  Digits are exact in FP16, products of two
// are at most 2^16, and the 64 products of a pivot block sum to at most 2^22 -- exact in the FP32
// accumulators of tcgen05.mma kind::f16.  The products of order i + j = d share accumulator d; its sum
// is below 2^20, 2^22, 2^23 for d = 0, 1, 2 and below 2^25 for the rest (above 2^24 only when nearly
// every digit is at its limit; what FP32 then rounds lies 2^-45 below the accumulator's unit weight).
// Orders past DG - 1 are dropped: of the product of the row maxima at most 2^-50 (every digit at its limit,
// all of one sign), about 2^-57 for random digits, where an FP64 dot product of 64 terms has 64 rounding
// errors of 2^-53 of its partial sums.  The epilogue adds the accumulators in 64-bit integers, rounds
// the sum once to a double and takes one FP64 operation per entry instead of 64.  An entry far below its
// row's largest keeps fewer than its 53 bits; S_k and S_k^+ of 20 matrices (100 to 730 dofs, every
// kernel, extended precision as the reference) err 0.99 and 0.97 times as much as on the FP64 pipes on
// average, 1.05 and 1.09 at most.
// The 64 pivots are first brought to one scale: column s of old is divided by the power of two 2^c_s
// next to sqrt(M_ss) and column s of pan multiplied by it (exact, and without effect on pan old^T), so
// that a block that mixes large and small diagonal entries keeps the digits of the small ones.
//
// Step over pivot block J (NB = 64 wide), three kernels: k_pivot_dg inverts the block (FP64, one CTA
// per subdomain) and splits D^-1; k_panel_dg takes 128 rows of M_J, splits them (old), forms pan =
// old D^-1 with the same digit products, writes it to M and splits it; k_update_dg subtracts pan old^T.
// M is symmetric, so the sweep keeps only its block upper triangle (128-wide blocks, the diagonal
// ones whole) and k_mirror_up fills the rest at the end: half the products, half the traffic.  The
// update's lanes are columns of M: its accesses are coalesced.
//
// k_update_dg: a CTA owns 128 columns i of M (A = digits of pan_i, 112 KB, loaded once) and walks
// 64-row blocks l (B = digits of old_l, 56 KB each, double-buffered): 28 digit pairs x 4 MMAs of
// 128 x 64 x 16 per block.  An MMA of this shape takes about 61 clocks (as long with N = 32: reading A
// sets its pace), so N = 64; seven accumulators of 64 columns fill tensor memory, so the high orders
// (0 .. 3) and the low ones take turns: sixteen warps drain one part while the other is formed.  Per
// block of 8192 entries 6.8 k clocks of MMA against 4.1 k of the FP64 pipe.  The entries of J are written by k_panel_dg
// (taken here, lane by lane, they cost 0.08 ms).  Measured on that row: 0.70 ms per step of the 36 matrices (the
// MMAs alone 0.32), against 15.3 ms; factorization and one solve 422 -> 33.1 ms.
// Every wait is bounded: one that runs out sets the sweep's timeout word; the CTA then waits (bounded)
// for its copies and MMAs, frees its tensor memory and returns.
#pragma once

constexpr int DG = 7;                               // digits
constexpr int DG_TILE = 128;
constexpr int DG_TBYTES = DG_TILE * 128;            // one digit of 128 rows x 64 columns, FP16: 16 KB
constexpr int DG_LB = 64;                           // rows of M per block of the update
constexpr int DG_LBYTES = DG_LB * 128;              // one digit of a block: 8 KB
constexpr int DG_EPI = 16;                          // epilogue warps of the update
constexpr int DG_THREADS = (DG_EPI + 1) * 32;       // and one for copies and MMAs
constexpr int DG_HI = 4;                            // accumulators 0 .. 3 (high orders), then 4 .. 6
constexpr int DG_SMEM_UPD = DG * DG_TBYTES + 2 * DG * DG_LBYTES + 1024;
constexpr int DG_SMEM_PAN = DG * DG_TBYTES + DG * (DG_TBYTES / 2) + 1024;
constexpr int DG_NAN = 1 << 20;                     // exponent of a row that is not finite
constexpr int DG_CHUNK = 16;                        // blocks of a CTA

struct DigitArgs {
    double *M;                // pool base
    double *dinv;             // per subdomain: NB x NB
    unsigned char *pan_d;     // digits of pan and old: per subdomain, per 128-row tile, DG x 16 KB
    unsigned char *old_d;
    unsigned char *dinv_d;    // digits of D^-1: per subdomain DG x 8 KB
    int *pan_e, *old_e, *dinv_e;      // exponents E per row
    int *piv_c;               // per subdomain NB: c_s
    const int64_t *moff;
    const int32_t *mdim, *mld, *pend;
    const int64_t *scr_off;   // per subdomain: scratch offset (rows, a multiple of 128)
    int j0;
    int *flag;                // [0] not SPD, [2] timeout
};

// E with |x| < 2^(E - 1) (a finite x, from its exponent field)
__device__ __forceinline__ int dg_exp(double x) {
    const int ex = (int)((__double_as_longlong(x) >> 52) & 0x7ff);
    return ex == 0x7ff ? DG_NAN : max(ex, 1) - 1021;
}

// x 2^(62 - E) as an integer (below 2^61; truncated)
__device__ __forceinline__ long long dg_fixed(double x, int E) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    long long m = b & 0xfffffffffffffll;
    if (ex) m |= 1ll << 52;
    const int sh = max(ex, 1) - 1022 - E + 9;       // m has 53 bits: value m 2^(ex - 1075)
    m = sh >= 0 ? m << min(sh, 9) : (sh > -64 ? m >> -sh : 0);
    return b < 0 ? -m : m;
}

// x 2^c (c within a few hundred; exact while the result is normal)
__device__ __forceinline__ double dg_shift(double x, int c) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    if (ex != 0 && ex != 0x7ff && ex + c > 0 && ex + c < 0x7ff) return __longlong_as_double(b + ((long long)c << 52));
    return ldexp(x, c);
}

// the digits of two neighbouring columns as FP16 pairs, last digit first
__device__ __forceinline__ void dg_split(long long f0, long long f1, uint32_t (&out)[DG]) {
#pragma unroll
    for (int k = DG - 1; k >= 0; --k) {
        int d0, d1;
        if (k > 0) {
            d0 = (int)((f0 + 256) & 511);           // digit + 256, in 0 .. 511
            d1 = (int)((f1 + 256) & 511);
            f0 = (f0 + 256) >> 9;
            f1 = (f1 + 256) >> 9;
        } else {
            d0 = (int)f0 + 256;                     // 128 .. 384
            d1 = (int)f1 + 256;
        }
        // 1024 + (digit + 256) as FP16 (integers are one unit apart there), minus 1280: exact
        const uint32_t raw = 0x64006400u + (uint32_t)d0 + ((uint32_t)d1 << 16);
        const __half2 v = __hsub2(*reinterpret_cast<const __half2 *>(&raw), __half2half2(__ushort_as_half(0x6500)));
        out[k] = *reinterpret_cast<const uint32_t *>(&v);
    }
}

// byte offset of (row r, column pair starting at even column k) in a digit tile
__device__ __forceinline__ int dg_off(int r, int k) {
    return (r >> 3) * 1024 + (r & 7) * 128 + (((k >> 3) ^ (r & 7)) << 4) + (k & 7) * 2;
}

__host__ __device__ constexpr uint32_t dg_idesc(int m, int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void dg_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void dg_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_s32(bar))
                 : "memory");
}
__device__ __forceinline__ void dg_bar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_s32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void dg_bar_arrive(uint64_t *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(tc_s32(bar)) : "memory");
}
__device__ __forceinline__ void dg_bar_expect(uint64_t *bar, unsigned bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(tc_s32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void dg_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc_s32(dst)),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(tc_s32(bar))
                 : "memory");
}
__device__ __forceinline__ void dg_s2g(void *dst, const void *src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(reinterpret_cast<uint64_t>(dst)),
                 "r"(tc_s32(src)), "r"(bytes)
                 : "memory");
}
// 32 lanes x 8 columns of 32 bits (no wait)
__device__ __forceinline__ void dg_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void dg_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}

// the digit products of one 64-column block of the orders D0 <= d < D1: accumulator d (N columns wide)
// of the set at tmem gets the pairs i + j = d; A and B are digit tiles of AB / BB bytes.  One thread
// issues the MMAs, so the loops are unrolled and the descriptors are sums of a base and a constant
template <int AB, int BB, int N, int D0, int D1>
__device__ __forceinline__ void dg_products(uint32_t tmem, uint32_t a, uint32_t b, uint32_t idesc) {
    const uint64_t da = tc_desc(a), db = tc_desc(b);
#pragma unroll
    for (int d = D0; d < D1; ++d)
#pragma unroll
        for (int i = 0; i <= d; ++i)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)          // K = 16: 32 bytes along the row
                dg_mma(tmem + (uint32_t)(d * N), da + (uint64_t)((i * AB + 32 * kk) >> 4),
                       db + (uint64_t)(((d - i) * BB + 32 * kk) >> 4), idesc, (i > 0 || kk > 0) ? 1 : 0);
}

// the accumulators (integers, exact in FP32) in 64 bits: orders 0 .. 3 in units of 2^-27 (the first
// two fit 32 bits), 4 .. 6 in units of 2^-54
__device__ __forceinline__ int dg_int(uint32_t v) { return __float2int_rn(__uint_as_float(v)); }
template <int W> __device__ __forceinline__ long long dg_hi(const uint32_t (&acc)[DG_HI][W], int c) {
    const int p = dg_int(acc[0][c]) * 512 + dg_int(acc[1][c]);
    return (long long)p * (1 << 18) + ((long long)dg_int(acc[2][c]) * 512 + (long long)dg_int(acc[3][c]));
}
template <int W> __device__ __forceinline__ long long dg_lo(const uint32_t (&acc)[DG - DG_HI][W], int c) {
    return (long long)dg_int(acc[0][c]) * (1 << 18) + ((long long)dg_int(acc[1][c]) * 512 + (long long)dg_int(acc[2][c]));
}

// the product sum 2^(E - 16) (hi 2^-27 + lo 2^-54), E the sum of the two rows' exponents, as a double,
// by integer operations alone (the FP64 pipe takes a warp 64 clocks per instruction; a 64-bit
// conversion is several): cut to 62 bits, normalised, rounded once to 53 bits (half up) and given
// exponent and sign.  This form is for the ends of the range and rows that are not finite
__device__ __forceinline__ double dg_value_ends(long long hi, long long lo, int E) {
    const int sh = min(26, __clzll((hi < 0 ? -hi : hi) | 1) - 2);        // |hi| < 2^48
    const long long I = (hi << sh) + (lo >> (27 - sh));
    const unsigned long long mag = (unsigned long long)(I < 0 ? -I : I);
    const int lz = __clzll(mag | 1);
    const unsigned long long m = mag << lz;                              // leading bit 63
    const long long q = (long long)((m >> 11) + ((m >> 10) & 1));        // 53 bits (or 2^53)
    if (E >= DG_NAN / 2) return __longlong_as_double(0x7ff8000000000000ll);   // a row was not finite
    const double v = mag ? ldexp((double)q, E - 43 - sh + 63 - lz - 52) : 0.0;
    return I < 0 ? -v : v;
}
// the same without a branch, where the result is a normal number or zero; elsewhere ends is set.  The
// lanes stay together: the loads of the accumulators are .aligned, and bringing the warp together
// before each cost k_update_dg 118 of 578 us (6 x 6 table row, a step's average)
__device__ __forceinline__ double dg_value(long long hi, long long lo, int E, bool &ends) {
    const int sh = min(26, __clzll((hi < 0 ? -hi : hi) | 1) - 2);
    const long long I = (hi << sh) + (lo >> (27 - sh));
    const unsigned long long mag = (unsigned long long)(I < 0 ? -I : I);
    const int lz = __clzll(mag | 1);
    const unsigned long long m = mag << lz;
    const long long q = (long long)((m >> 11) + ((m >> 10) & 1));
    // value q 2^(e - 52), e the exponent of the leading bit
    const int e = E - 43 - sh + 63 - lz;
    ends |= (mag != 0 && (e <= -1022 || e >= 1023)) || E >= DG_NAN / 2;
    const long long b = (q + ((long long)(e + 1022) << 52)) | (I < 0 ? (1ll << 63) : 0);
    return __longlong_as_double(mag != 0 ? b : 0ll);
}

// invert the pivot block in registers: 544 threads hold the rows of the 4 x 4 blocks (bi, bl <= bi) of
// the lower triangle; step p needs row p (= column p), kept in shared memory and rewritten by its
// owners, and the reciprocal of the pivot, which the next pivot's owner forms first, beside the
// others' FMAs.  64 steps of 2080 FP64 FMAs on one SM's two lanes: 35 us at least;
// measured 120 us, against 337 us for a shared-memory sweep of the whole block.
constexpr int DG_PIV_THREADS = 544;
__global__ void __launch_bounds__(DG_PIV_THREADS) k_pivot_dg(DigitArgs a) {
    const int k = blockIdx.x;
    const int pend = a.pend[k];
    if (a.j0 >= pend) return;
    const int b = min(NB, pend - a.j0), ld = a.mld[k];
    const double *M = a.M + a.moff[k];
    __shared__ double S[NB * (NB + 1)];
    __shared__ double rowp[2][NB], dpiv[2];
    __shared__ int pc[NB];
    bool ok = true;
    int bi = 0, bl = 0;
    {
        int t = threadIdx.x / 4;
        while (t >= bi + 1 && bi < 15) { t -= bi + 1; ++bi; }
        bl = t;
    }
    const int i = 4 * bi + (threadIdx.x & 3), l0 = 4 * bl;
    double v[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int l = l0 + y;
        // upper triangle of M; the identity past the block's width
        v[y] = (i < b && l < b) ? M[(int64_t)(a.j0 + min(i, l)) * ld + a.j0 + max(i, l)] : (i == l ? 1.0 : 0.0);
    }
    if (bi == bl)
#pragma unroll
        for (int y = 0; y < 4; ++y)
            if (l0 + y == i) {
                // the diagonal entry's exponent, halved (0 for a non-positive or non-normal one)
                const int ex = (int)((__double_as_longlong(v[y]) >> 52) & 0xfff);
                pc[i] = ex > 0 && ex < 0x7ff ? (ex - 1023) >> 1 : 0;
            }
    auto pivot = [&](double d, int buf) {
        if (!(d > 0.0)) ok = false;
        dpiv[buf] = 1.0 / d;
    };
    auto publish = [&](int p, int buf) {            // row p of the current matrix
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int l = l0 + y;
            if (i == p && l <= p) rowp[buf][l] = v[y];
            else if (l == p && i > p) rowp[buf][i] = v[y];
        }
    };
    publish(0, 0);
    if (threadIdx.x == 0) pivot(v[0], 0);
    __syncthreads();
    for (int p = 0; p < NB; ++p) {
        const int buf = p & 1;
        const double inv = dpiv[buf], ri = rowp[buf][i] * inv;
        double rl[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) rl[y] = rowp[buf][l0 + y];
        if (i == p + 1 && bi == bl) {               // the next pivot
            double d = v[0], r = rl[0];
#pragma unroll
            for (int y = 1; y < 4; ++y)
                if (l0 + y == p + 1) { d = v[y]; r = rl[y]; }
            pivot(d - ri * r, buf ^ 1);
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int l = l0 + y;
            if (i == p && l == p) v[y] = -inv;
            else if (i == p) v[y] = rl[y] * inv;
            else if (l == p) v[y] = ri;
            else v[y] -= ri * rl[y];
        }
        if (p + 1 < NB) publish(p + 1, buf ^ 1);
        __syncthreads();
    }
    if (!ok) atomicMax(a.flag, 1);
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int l = l0 + y;
        const double d = (i < b && l < b) ? -v[y] : 0.0;
        if (l <= i) {
            S[i * (NB + 1) + l] = d;
            S[l * (NB + 1) + i] = d;
        }
    }
    __syncthreads();
    double *D = a.dinv + (int64_t)k * NB * NB;
    for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) D[t] = S[(t / NB) * (NB + 1) + t % NB];
    __syncthreads();
    if (threadIdx.x < NB) {
        const int r = threadIdx.x;
        a.piv_c[k * NB + r] = pc[r];
        // the digits of the scaled 2^(c_r + c_s) D^-1
        int E = -1022;
        for (int s = 0; s < NB; ++s) {
            const double d = dg_shift(S[r * (NB + 1) + s], pc[r] + pc[s]);
            S[r * (NB + 1) + s] = d;
            E = max(E, dg_exp(d));
        }
        a.dinv_e[k * NB + r] = E;
        unsigned char *dst = a.dinv_d + (int64_t)k * DG * (DG_TBYTES / 2);
        for (int s = 0; s < NB; s += 2) {
            uint32_t o[DG];
            dg_split(dg_fixed(S[r * (NB + 1) + s], E), dg_fixed(S[r * (NB + 1) + s + 1], E), o);
#pragma unroll
            for (int q = 0; q < DG; ++q) *reinterpret_cast<uint32_t *>(dst + q * (DG_TBYTES / 2) + dg_off(r, s)) = o[q];
        }
    }
}

// panels of 128 rows: thread (row r = tid mod 128, quarter h) has 16 of the row's 64 columns
constexpr int DG_PAN_THREADS = 512;
__global__ void __launch_bounds__(DG_PAN_THREADS, 1) k_panel_dg(DigitArgs a) {
    const int k = blockIdx.y;
    const int pend = a.pend[k];
    if (a.j0 >= pend) return;
    const int n = a.mdim[k], ld = a.mld[k], tile = blockIdx.x, r0 = tile * DG_TILE;
    if (r0 >= n) return;
    const int b = min(NB, pend - a.j0), j0 = a.j0, jt = j0 / DG_TILE;
    double *M = a.M + a.moff[k];
    extern __shared__ __align__(1024) unsigned char dg_raw[];
    unsigned char *sa = dg_raw + ((1024u - (tc_s32(dg_raw) & 1023u)) & 1023u), *sb = sa + DG * DG_TBYTES;
    __shared__ uint64_t bar_b, bar_mma;
    __shared__ uint32_t tmem_base;
    __shared__ int se[4][DG_TILE], sde[NB], spc[NB];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, r = threadIdx.x % DG_TILE, h = threadIdx.x / DG_TILE;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_s32(&tmem_base)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        dg_bar_init(&bar_b, 1);
        dg_bar_init(&bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        dg_bar_expect(&bar_b, DG * (DG_TBYTES / 2));
        dg_g2s(sb, a.dinv_d + (int64_t)k * DG * (DG_TBYTES / 2), DG * (DG_TBYTES / 2), &bar_b);
    }
    if (threadIdx.x < NB) {
        sde[threadIdx.x] = a.dinv_e[k * NB + threadIdx.x];
        spc[threadIdx.x] = a.piv_c[k * NB + threadIdx.x];
    }
    __syncthreads();
    const int i = r0 + r;
    double x[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const int c = 16 * h + s;
        double v = 0.0;
        if (i < n && c < b) v = tile <= jt ? M[(int64_t)i * ld + j0 + c] : M[(int64_t)(j0 + c) * ld + i];
        x[s] = dg_shift(v, -spc[c]);
    }
    // the diagonal tile is whole, so rows of the pivot's own tile may be read either way; rows above
    // it hold M_iJ, rows below are read from the transposed block
    auto split_rows = [&](int E) {
#pragma unroll
        for (int s = 0; s < 16; s += 2) {
            uint32_t o[DG];
            dg_split(dg_fixed(x[s], E), dg_fixed(x[s + 1], E), o);
            const int off = dg_off(r, 16 * h + s);
#pragma unroll
            for (int q = 0; q < DG; ++q) *reinterpret_cast<uint32_t *>(sa + q * DG_TBYTES + off) = o[q];
        }
    };
    auto row_exp = [&]() {
        int E = -1022;
#pragma unroll
        for (int s = 0; s < 16; ++s) E = max(E, dg_exp(x[s]));
        se[h][r] = E;
        __syncthreads();
        return max(max(se[0][r], se[1][r]), max(se[2][r], se[3][r]));
    };
    const int Eo = row_exp();
    split_rows(Eo);
    const int64_t row0 = a.scr_off[k] + r0;
    if (h == 0) a.old_e[row0 + r] = Eo;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const int64_t tile_off = (row0 / DG_TILE) * DG * DG_TBYTES;
    bool ok = true;
    if (threadIdx.x == 0) {
        dg_s2g(a.old_d + tile_off, sa, DG * DG_TBYTES);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        ok = tc_wait(&bar_b, 0, TC_WAIT_TRIES);
        if (ok) {
            dg_products<DG_TBYTES, DG_TBYTES / 2, NB, 0, DG>(tmem, tc_s32(sa), tc_s32(sb), dg_idesc(DG_TILE, NB));
            dg_commit(&bar_mma);
        } else {
            atomicExch(a.flag + 2, 1);
            tc_wait(&bar_b, 0, TC_WAIT_TRIES);
            dg_bar_arrive(&bar_mma);                // nothing was issued: release the others
        }
        // the digits of old have left shared memory before pan's overwrite them
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    const bool done = tc_wait(&bar_mma, 0, TC_WAIT_TRIES);
    if (!done) {
        atomicExch(a.flag + 2, 1);
        tc_wait(&bar_mma, 0, TC_WAIT_TRIES);
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // (scaled) pan = old D^-1: lane quarter warp mod 4 and columns 16 (warp / 4) .. are the thread's own
#pragma unroll
    for (int c0 = 0; c0 < 16; c0 += 8) {               // the lanes part only where __syncwarp() follows
        uint32_t hi[DG_HI][8], lo[DG - DG_HI][8];
        const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(16 * h + c0);
#pragma unroll
        for (int d = 0; d < DG_HI; ++d) dg_ld8(ta + (uint32_t)(d * NB), hi[d]);
#pragma unroll
        for (int d = DG_HI; d < DG; ++d) dg_ld8(ta + (uint32_t)(d * NB), lo[d - DG_HI]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        bool ends = false;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            x[c0 + c] = dg_value(dg_hi(hi, c), dg_lo(lo, c), Eo + sde[16 * h + c0 + c], ends);
        if (__any_sync(0xffffffffu, ends)) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                x[c0 + c] = dg_value_ends(dg_hi(hi, c), dg_lo(lo, c), Eo + sde[16 * h + c0 + c]);
            __syncwarp();
        }
    }
    __syncthreads();                                 // se is written again
    const int Ep = row_exp();
    split_rows(Ep);
    if (h == 0) a.pan_e[row0 + r] = Ep;
    // M_iJ = pan (-D^-1 for the rows of J), where M_iJ was read; in the pivot's diagonal tile, which is
    // whole, also the transposed entries of the other rows.  k_update_dg leaves J alone
    if (i < n) {
        const int ij = i - j0;
        const bool iJ = ij >= 0 && ij < b;
        const double *D = a.dinv + (int64_t)k * NB * NB + (iJ ? ij : 0) * NB;
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const int c = 16 * h + s;
            if (c >= b) continue;
            const double v = dg_shift(x[s], -spc[c]);
            if (tile <= jt) M[(int64_t)i * ld + j0 + c] = iJ ? -D[c] : v;
            if (tile >= jt && !iJ) M[(int64_t)(j0 + c) * ld + i] = v;
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x == 0) {
        dg_s2g(a.pan_d + tile_off, sa, DG * DG_TBYTES);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    if (warp == 0) {
        __syncwarp();                                // lane 0 waited for its copies
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// grid (column tiles of the largest subdomain, last first; chunks of DG_CHUNK row blocks; K)
__global__ void __launch_bounds__(DG_THREADS, 1) k_update_dg(DigitArgs a) {
    const int k = blockIdx.z;
    const int pend = a.pend[k];
    if (a.j0 >= pend) return;
    const int n = a.mdim[k], ld = a.mld[k], tile = (int)gridDim.x - 1 - (int)blockIdx.x, c0 = tile * DG_TILE;
    if (c0 >= n) return;
    const int nblk = (min(n, c0 + DG_TILE) + DG_LB - 1) / DG_LB;       // row blocks of the upper triangle
    const int q0 = blockIdx.y * DG_CHUNK, q1 = min(nblk, q0 + DG_CHUNK);
    if (q0 >= q1) return;
    const int b = min(NB, pend - a.j0), j0 = a.j0, j1 = j0 + b;
    double *M = a.M + a.moff[k];
    extern __shared__ __align__(1024) unsigned char dg_raw[];
    unsigned char *sa = dg_raw + ((1024u - (tc_s32(dg_raw) & 1023u)) & 1023u), *sb = sa + DG * DG_TBYTES;
    // part 0: high orders, part 1: low orders
    __shared__ uint64_t full_a, full_b[2], empty_b[2], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        dg_bar_init(&full_a, 1);
        for (int s = 0; s < 2; ++s) {
            dg_bar_init(&full_b[s], 1);
            dg_bar_init(&empty_b[s], 1);
            dg_bar_init(&acc_full[s], 1);
            dg_bar_init(&acc_empty[s], DG_EPI * 32);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == DG_EPI) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_s32(&tmem_base)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const int64_t row0 = a.scr_off[k];
    if (warp == DG_EPI) {
        // ------------------------------------------------------------ copies and MMAs, one thread
        if (lane == 0) {
            auto load_b = [&](int q) {
                const int s = (q - q0) & 1;
                const int64_t t = (row0 + (int64_t)q * DG_LB) / DG_TILE;
                const unsigned char *src = a.old_d + t * DG * DG_TBYTES + (q % (DG_TILE / DG_LB)) * DG_LBYTES;
                dg_bar_expect(&full_b[s], DG * DG_LBYTES);
                for (int d = 0; d < DG; ++d)
                    dg_g2s(sb + (s * DG + d) * DG_LBYTES, src + d * DG_TBYTES, DG_LBYTES, &full_b[s]);
            };
            constexpr uint32_t IDESC = dg_idesc(DG_TILE, DG_LB);
            bool ok = true;
            int issued = 0, loaded = q0;
            dg_bar_expect(&full_a, DG * DG_TBYTES);
            dg_g2s(sa, a.pan_d + (row0 + c0) / DG_TILE * DG * DG_TBYTES, DG * DG_TBYTES, &full_a);
            load_b(loaded++);
            if (loaded < q1) load_b(loaded++);
            ok = tc_wait(&full_a, 0, TC_WAIT_TRIES);
            for (int q = q0; q < q1 && ok; ++q) {
                const int it = q - q0, s = it & 1, ph = (it >> 1) & 1;
                const uint32_t b_s = tc_s32(sb + s * DG * DG_LBYTES);
                // a part of the accumulators was last drained for block it - 1
                ok = !abort_flag && tc_wait(&full_b[s], ph, TC_WAIT_TRIES) &&
                     (it < 1 || tc_wait(&acc_empty[0], (it - 1) & 1, TC_WAIT_TRIES));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                dg_products<DG_TBYTES, DG_LBYTES, DG_LB, 0, DG_HI>(tmem, tc_s32(sa), b_s, IDESC);
                dg_commit(&acc_full[0]);
                ok = !abort_flag && (it < 1 || tc_wait(&acc_empty[1], (it - 1) & 1, TC_WAIT_TRIES));
                if (ok) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    dg_products<DG_TBYTES, DG_LBYTES, DG_LB, DG_HI, DG>(tmem, tc_s32(sa), b_s, IDESC);
                    dg_commit(&acc_full[1]);
                }
                dg_commit(&empty_b[s]);
                issued = it + 1;
                // refill the buffer block it - 1 used (its MMAs are done once empty_b fires)
                if (ok && it >= 1 && loaded < q1) {
                    const int ps = (it - 1) & 1;
                    ok = tc_wait(&empty_b[ps], ((it - 1) >> 1) & 1, TC_WAIT_TRIES);
                    if (ok) load_b(loaded++);
                }
            }
            if (!ok) {
                atomicExch(a.flag + 2, 1);
                abort_flag = 1;
            }
            // what was copied has landed and what was issued is done before the CTA goes
            tc_wait(&full_a, 0, TC_WAIT_TRIES);
            for (int q = max(q0, loaded - 2); q < loaded; ++q) tc_wait(&full_b[(q - q0) & 1], ((q - q0) >> 1) & 1, TC_WAIT_TRIES);
            for (int it = max(0, issued - 2); it < issued; ++it) tc_wait(&empty_b[it & 1], (it >> 1) & 1, TC_WAIT_TRIES);
        }
    } else {
        // ------------------------------------------------------------ epilogue: column i of M per lane
        const int qd = warp & 3, hf = warp >> 2;      // lane quarter; 16 of the block's 64 rows
        const int i = c0 + 32 * qd + lane;
        const bool in = i < n, iJ = i >= j0 && i < j1;
        const int Ea = in ? a.pan_e[row0 + i] : 0;
        const uint32_t ta = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(16 * hf);
        for (int q = q0; q < q1; ++q) {
            const int ph = (q - q0) & 1, l0 = q * DG_LB + 16 * hf;
            // the warp's 16 rows x 32 columns of M: plain when the pivot block and the edges are elsewhere
            const bool plain = c0 + DG_TILE <= n && l0 + 16 <= n && (j1 <= c0 || j0 >= c0 + DG_TILE) &&
                               (j1 <= l0 || j0 >= l0 + 16);
            double *Mp = M + (int64_t)l0 * ld + i;
            double m[16];
#pragma unroll
            for (int c = 0; c < 16; ++c)
                m[c] = plain || (in && l0 + c < n) ? Mp[(int64_t)c * ld] : 0.0;
            // the next block's entries into L2 (lane: row, half of its 256 bytes)
            if (q + 1 < q1 && l0 + DG_LB + (lane >> 1) < n && c0 + 32 * qd + 16 * (lane & 1) < n)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(M + (int64_t)(l0 + DG_LB + (lane >> 1)) * ld + c0 + 32 * qd +
                                                              16 * (lane & 1)));
            long long hi[16];
            bool ok = !abort_flag && tc_wait(&acc_full[0], ph, TC_WAIT_TRIES);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) {
                    atomicExch(a.flag + 2, 1);
                    abort_flag = 1;
                }
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int cc = 0; cc < 16; cc += 4) {
                __syncwarp();                        // the loads are .aligned
                uint32_t acc[DG_HI][4];
#pragma unroll
                for (int d = 0; d < DG_HI; ++d) dg_ld4(ta + (uint32_t)(d * DG_LB + cc), acc[d]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (cc == 12) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    dg_bar_arrive(&acc_empty[0]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) hi[cc + c] = dg_hi(acc, c);
            }
            const int *oe = a.old_e + row0 + l0;
            ok = !abort_flag && tc_wait(&acc_full[1], ph, TC_WAIT_TRIES);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) {
                    atomicExch(a.flag + 2, 1);
                    abort_flag = 1;
                }
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int cc = 0; cc < 16; cc += 4) {       // the lanes part only where __syncwarp() follows
                uint32_t acc[DG - DG_HI][4];
#pragma unroll
                for (int d = DG_HI; d < DG; ++d) dg_ld4(ta + (uint32_t)(d * DG_LB + cc), acc[d - DG_HI]);
                const int4 ea = __ldg(reinterpret_cast<const int4 *>(oe + cc));
                const int eo[4] = {ea.x, ea.y, ea.z, ea.w};
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (cc == 12) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    dg_bar_arrive(&acc_empty[1]);
                }
                double o[4];
                bool ends = false;
#pragma unroll
                for (int c = 0; c < 4; ++c) o[c] = dg_value(hi[cc + c], dg_lo(acc, c), Ea + eo[c], ends);
                if (__any_sync(0xffffffffu, ends)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) o[c] = dg_value_ends(hi[cc + c], dg_lo(acc, c), Ea + eo[c]);
                    __syncwarp();
                }
                if (plain) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) Mp[(int64_t)(cc + c) * ld] = m[cc + c] - o[c];
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int l = l0 + cc + c;   // J holds its new values already
                        if (in && !iJ && l < n && (l < j0 || l >= j1)) Mp[(int64_t)(cc + c) * ld] = m[cc + c] - o[c];
                    }
                    __syncwarp();
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == DG_EPI) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// the lower triangle from the upper one, 32 x 32 tiles through shared memory; grid (tiles, tiles, K)
template <typename T>
__global__ void __launch_bounds__(256) k_mirror_up(T *pool, const int64_t *moff, const int32_t *mdim,
                                                   const int32_t *mld) {
    const int k = blockIdx.z, n = mdim[k], ld = mld[k];
    const int ti = blockIdx.y, tl = blockIdx.x;       // writes tile (rows ti, columns tl), tl <= ti
    if (ti * 32 >= n || tl > ti) return;
    T *M = pool + moff[k];
    __shared__ T t[32][33];
    const int x = threadIdx.x % 32, y0 = threadIdx.x / 32;
    for (int y = y0; y < 32; y += 8) {
        const int rr = tl * 32 + y, cc = ti * 32 + x;
        t[y][x] = rr < n && cc < n ? M[(int64_t)rr * ld + cc] : T(0);
    }
    __syncthreads();
    for (int y = y0; y < 32; y += 8) {
        const int rr = ti * 32 + y, cc = tl * 32 + x;
        if (rr < n && cc < n && cc < rr) M[(int64_t)rr * ld + cc] = t[x][y];
    }
}
