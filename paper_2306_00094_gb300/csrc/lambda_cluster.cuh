// Lambda-space work of a PCG iteration as two kernels, one thread-block cluster per group of
// right-hand sides.
//
// Between the two interface applies of an iteration lie chains of short steps, each needing a sum
// over all Lambda rows before the next can start:
//   k_lam_a (after S^+):  q = B y_U, (p, q), eta;  G^T r_new, alpha;  p, lambda, r, w = P r, (w, w),
//                         stop test;  x = B_D^T w;
//   k_lam_b (after S):    z = B_D y_U;  G^T z, alpha;  y = P z, (y, w), beta;  x = B^T p_new.
// As one kernel per step (lambda_rows.cuh) they are latency-bound: a launch with a fused reduction takes 7-10 us even
// on a few hundred rows (start-up, fence, arrival atomic, the last block's finish), where the data
// (a few MB, resident in L2) would take one or two.  The right-hand sides of a PCG are independent
// of one another, so a cluster of LC CTAs (16 SMs of one GPC) owns CW of them for the whole kernel,
// the steps are separated by the cluster's hardware barrier, and the sums travel through distributed
// shared memory: every CTA sends its partials to all others and every CTA forms the same totals and
// scalars, so a reduction costs one barrier.  The clusters never wait for one another.
// Measured (ncu, warm caches, one iteration's Lambda work; cluster kernels against one kernel per
// step): 309 rows x 1: 9.8 + 6.6 us against 43; 13455 rows x 8: 20.1 + 12.8 against 55.5.  One
// cluster per pair of columns reads every index once per pair, so its SMs' load units set the pace
// when a thread has several rows: 38150 rows x 16: 62 + 45 us against 90.  So the line lies at one
// row per thread (LAM_MAX_ROWS); problems past it keep the kernels per step.  It depends on n_lambda
// alone: the sums of the two forms are ordered differently, and a column must not notice its batch.
//
// Layout: the PCG vectors are kept per group, row by row with the CW columns consecutive (entry
// (i, c) of group g at (g n + i) CW + c), so that a group's loads are dense; columns past R are
// zeros that nothing activates.  B, B_D, their transposes and G = B Z are read in ELL form (entry e
// of row i at e n + i, int32, -1 past the row's end), built once per problem: no row pointers, and
// coalesced.
//
// Order of the sums: a thread's rows, lanes and CTAs follow from n alone (CTA rank, thread, then
// stride LC LAM_THREADS), so a column's result does not depend on the batch it is part of or on CW.
// Dot products: products in L; the FP32 sums of a thread and of 4 lanes are compensated (TwoSum), the
// rest FP64.
#pragma once



constexpr int LC = 16;                     // CTAs of a cluster (non-portable size)
constexpr int LAM_THREADS = 1024;
constexpr int LAM_WARPS = LAM_THREADS / 32;
constexpr int LAM_MAX_ELL = 16;            // entries per row of B_D and B_D^T (copies of a node)
constexpr int LAM_MAX_CO = 2048;           // coarse columns (shared memory)
constexpr int64_t LAM_MAX_ROWS = LC * LAM_THREADS;   // Lambda rows: one per thread
constexpr size_t LAM_MAX_SMEM = 192 * 1024;
constexpr int LAM_CO_ALL = 128;            // FP32: n_co up to which every CTA solves for all of alpha
constexpr int LAM_PARTS = 8;               // the sum over j of a row of (G^T G)^-1 in this many parts

// columns per cluster for R right-hand sides: one for one; pairs while the clusters of a launch fit
// on the device at once (one per GPC), else four
__host__ __device__ inline int lam_cw(int R, int elem_size) {
    return R == 1 ? 1 : (R <= 16 || elem_size == 8 ? 2 : 4);
}
// columns of the grouped layout: R rounded up to whole groups
__host__ __device__ inline int lam_rp(int R) {
    const int cw = lam_cw(R, 4);
    return (R + cw - 1) / cw * cw;
}
// slices of a floating subdomain's G^T sum (one warp each), from the number of floating subdomains
__host__ __device__ inline int lam_slices(int nf) { return nf <= 128 ? 8 : (nf <= 512 ? 2 : 1); }

template <typename L, int CW> struct alignas(sizeof(L) * CW) Pack { L v[CW]; };

template <typename L> struct LamArgs {
    // operators (ELL, int32 indices; values in L)
    const int32_t *bpm;                    // 2 x nl: U index of +1, of -1
    const int32_t *bt;                     // 2 x nu: signed rows r + 1 / -(r + 1), 0 = none
    const int32_t *bd_col;  const L *bd_val;    int bd_w;      // bd_w x nl
    const int32_t *bdt_row; const L *bdt_val;   int bdt_w;     // bdt_w x nu
    const int32_t *g_col;   const L *g_val;     int g_w;       // g_w x nl: first half +1 side, second -1 side
    const int32_t *gt_row;  const L *gt_w;      int64_t gt_n;  // B^T entries: Lambda row, 3 x gt_n weights
    const int64_t *gt_range; const int32_t *gt_co; int nf;
    const double *ginv;                    // (G^T G)^-1
    const float *ginv32;                   // its FP32 copy, transposed
    int nco;
    const int4 *u2x;                       // per U dof: place in the apply input
    // vectors
    const L *yU;                           // nu x R, interleaved
    L *r, *w, *z, *y, *pv, *q, *lam;       // grouped
    L *x;                                  // apply input (FP32: paired; FP64: columns)
    __half *x16;                           // set: the FP16 input of the tensor-core apply instead (k_lam_a)
    int nl, nu, R;
    PcgScalars s;
    double tol;
    int max_it, limit;
    cudaGraphConditionalHandle cond;
};

// a pack written by another CTA of the cluster in the same kernel: read at L2
template <typename L, int CW> __device__ __forceinline__ Pack<L, CW> ld_cg(const Pack<L, CW> *p) {
    Pack<L, CW> o;
    if constexpr (sizeof(L) == 4 && CW == 1) o.v[0] = __ldcg(&p->v[0]);
    else if constexpr (sizeof(L) == 4 && CW == 2) {
        const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
        o.v[0] = t.x; o.v[1] = t.y;
    } else if constexpr (sizeof(L) == 4) {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
        o.v[0] = t.x; o.v[1] = t.y; o.v[2] = t.z; o.v[3] = t.w;
    } else {
#pragma unroll
        for (int c = 0; c < CW; ++c) o.v[c] = __ldcg(&p->v[c]);
    }
    return o;
}

template <int CW> __device__ __forceinline__ bool act_of(const bool (&act)[CW], int c) {
    bool r = false;
#pragma unroll
    for (int k = 0; k < CW; ++k) r = k == c ? act[k] : r;
    return r;
}

// two-term sums: s + e with e the rounding errors of the additions (FP64: plain)
__device__ __forceinline__ void two_add(float &s, float &e, float v, float ve) {
    const float t = __fadd_rn(s, v), bb = __fsub_rn(t, s);
    e = __fadd_rn(__fadd_rn(e, ve), __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(v, bb)));
    s = t;
}
__device__ __forceinline__ void two_add(double &s, double &, double v, double) { s += v; }

// dynamic shared memory: gpart (n_co slices CW), g (n_co CW; FP64 for small n_co), alpha (n_co CW),
// parts
template <typename L, int CW> __host__ __device__ inline size_t lam_smem_bytes(int nco, int nf) {
    return sizeof(double) * (size_t)nco * CW + sizeof(L) * ((size_t)nco * lam_slices(nf) * CW + (size_t)nco * CW) +
           sizeof(L) * LAM_PARTS * 128 * CW;
}

// static shared memory of a kernel; the arrays that other CTAs write are used once per kernel each
template <typename L, int CW> struct LamShared {
    float2 unit[LAM_THREADS / 4][CW];      // sums of 4 lanes (FP32)
    double dunit[LAM_THREADS / 4][CW];     // the same (FP64)
    double part[2][LC][CW];                // per reduction: every CTA's partial (written by all CTAs)
    double yw_old[CW], xs[CW];             // scalars of the columns
    L step[CW], xsl[CW];                   // eta (k_lam_a) or beta (k_lam_b); the FP16 scale
    int on[CW], it[CW];
};

// every CTA of the cluster has started (needed once before the first access to another CTA's
// shared memory): arrive early, wait late
__device__ __forceinline__ void cluster_started_arrive() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_started_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// the cluster's sums of CW values per thread (s, e): this CTA's partial to every CTA's part[which],
// the cluster barrier, then fin(c, total) once per column in every CTA (one thread each: FP64
// divisions and roots by every thread would keep the FP64 pipe, 1/64 of the FP32 rate, busy for
// microseconds); what fin writes to shared memory is visible to the CTA afterwards
template <typename L, int CW, typename F>
__device__ __forceinline__ void cluster_sum(LamShared<L, CW> &sh, int which, L (&s)[CW], L (&e)[CW], F &&fin) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
#pragma unroll
    for (int o = 1; o <= 2; o *= 2)
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            const L vs = __shfl_xor_sync(0xffffffffu, s[c], o), ve = __shfl_xor_sync(0xffffffffu, e[c], o);
            // the same operands in the same order in both lanes
            L a = (lane & o) ? vs : s[c], ae = (lane & o) ? ve : e[c];
            const L b = (lane & o) ? s[c] : vs, be = (lane & o) ? e[c] : ve;
            two_add(a, ae, b, be);
            s[c] = a;
            e[c] = ae;
        }
    if ((lane & 3) == 0)
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            if constexpr (std::is_same<L, float>::value) sh.unit[threadIdx.x / 4][c] = make_float2(s[c], e[c]);
            else sh.dunit[threadIdx.x / 4][c] = s[c];
        }
    __syncthreads();
    if (warp < CW) {
        double v = 0;
#pragma unroll
        for (int k = 0; k < LAM_THREADS / 128; ++k) {
            if constexpr (std::is_same<L, float>::value) {
                const float2 f = sh.unit[lane + 32 * k][warp];
                v += (double)f.x + (double)f.y;
            } else {
                v += sh.dunit[lane + 32 * k][warp];
            }
        }
        v = warp_sum(v);
        if (lane < LC) *cl.map_shared_rank(&sh.part[which][cl.block_rank()][warp], lane) = v;
    }
    __syncwarp();
    cl.sync();
    if (warp < CW) {
        double v = lane < LC ? sh.part[which][lane][warp] : 0.0;
        v = warp_sum(v);
        if (lane == 0) fin(warp, v);
    }
    __syncthreads();
}

// alpha = (G^T G)^-1 G^T v for the group's columns into al (every CTA), v given per Lambda row by
// f(row) (a Pack); contains cluster barriers, so every thread of the cluster calls it
template <typename L, int CW, typename F>
__device__ __forceinline__ void cluster_alpha(const LamArgs<L> &a, unsigned char *dyn, L *&al, F &&f) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int ns = lam_slices(a.nf), nco = a.nco;
    double *g = reinterpret_cast<double *>(dyn);
    L *gpart = reinterpret_cast<L *>(g + (size_t)nco * CW);
    al = gpart + (size_t)nco * ns * CW;
    L *parts = al + (size_t)nco * CW;
    // one warp per (floating subdomain, slice): lanes over the entries, LAM_U in flight
    constexpr int LAM_U = 4;
    for (int un = rank * LAM_WARPS + warp; un < a.nf * ns; un += LC * LAM_WARPS) {
        const int fl = un / ns, sl = un % ns;
        const int64_t e0 = a.gt_range[4 * fl], e1 = a.gt_range[4 * fl + 1], ch = (e1 - e0 + ns - 1) / ns;
        const int64_t b0 = e0 + sl * ch, b1 = min(e1, b0 + ch);
        const int co = a.gt_co[2 * fl], nq = a.gt_co[2 * fl + 1];
        L acc[3][CW];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int c = 0; c < CW; ++c) acc[q][c] = L(0);
        for (int64_t b = b0 + lane; b < b1; b += 32 * LAM_U) {
            int row[LAM_U];
            Pack<L, CW> v[LAM_U];
#pragma unroll
            for (int u = 0; u < LAM_U; ++u) row[u] = b + 32 * u < b1 ? a.gt_row[b + 32 * u] : -1;
#pragma unroll
            for (int u = 0; u < LAM_U; ++u)
                if (row[u] >= 0) v[u] = f(row[u]);
#pragma unroll
            for (int u = 0; u < LAM_U; ++u)
                if (row[u] >= 0)
                    for (int q = 0; q < nq; ++q) {
                        const L w = a.gt_w[q * a.gt_n + b + 32 * u];
#pragma unroll
                        for (int qq = 0; qq < 3; ++qq)
                            if (qq == q)
#pragma unroll
                                for (int c = 0; c < CW; ++c) acc[qq][c] += w * v[u].v[c];
                    }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (q < nq)
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    const L t = warp_sum(acc[q][c]);
                    if (lane < LC) *cl.map_shared_rank(gpart + ((size_t)(co + q) * ns + sl) * CW + c, lane) = t;
                }
    }
    __syncwarp();
    cl.sync();
    const bool small = nco <= kCoarseFusedMax;
    L *gl = reinterpret_cast<L *>(g);
    for (int t = threadIdx.x; t < nco * CW; t += LAM_THREADS) {
        const int j = t / CW, c = t % CW;
        if (small) {
            double v = 0;
            for (int s = 0; s < ns; ++s) v += (double)gpart[((size_t)j * ns + s) * CW + c];
            g[t] = v;
        } else {
            L v = 0, ve = 0;
            for (int s = 0; s < ns; ++s) two_add(v, ve, gpart[((size_t)j * ns + s) * CW + c], L(0));
            gl[t] = v + ve;
        }
    }
    __syncthreads();
    if (small) {
        // FP64, one thread per (row, column)
        for (int t = threadIdx.x; t < nco * CW; t += LAM_THREADS) {
            const int i = t / CW, c = t % CW;
            double v = 0;
            for (int j = 0; j < nco; ++j) v += a.ginv[i * nco + j] * g[j * CW + c];
            al[t] = (L)v;
        }
        __syncthreads();
        return;
    }
    // rows [i0, i1) of this CTA: all of them (every CTA alike), or a 1/LC share sent to the others
    constexpr bool F32 = std::is_same<L, float>::value;
    const bool share = !F32 || nco > LAM_CO_ALL;
    const int chunk = share ? (nco + LC - 1) / LC : nco;
    const int i0 = share ? rank * chunk : 0, i1 = min(nco, i0 + chunk);
    const int pt = threadIdx.x / 128, il = threadIdx.x % 128, jc = (nco + LAM_PARTS - 1) / LAM_PARTS;
    {
        const int i = i0 + il;
        L acc[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = L(0);
        if (i < i1) {
            const int j1 = min(nco, (pt + 1) * jc);
#pragma unroll 8
            for (int j = pt * jc; j < j1; ++j) {
                L m;
                if constexpr (F32) m = __ldg(a.ginv32 + (size_t)j * nco + i);
                else m = __ldg(a.ginv + (size_t)j * nco + i);      // symmetric
#pragma unroll
                for (int c = 0; c < CW; ++c) acc[c] = fma_l(m, gl[j * CW + c], acc[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < CW; ++c) parts[(pt * 128 + il) * CW + c] = acc[c];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < (i1 - i0) * CW; t += LAM_THREADS) {
        L v = parts[t];
        for (int k = 1; k < LAM_PARTS; ++k) v += parts[k * 128 * CW + t];
        if (share)
            for (int rk = 0; rk < LC; ++rk) *cl.map_shared_rank(al + (size_t)i0 * CW + t, rk) = v;
        else al[t] = v;
    }
    __syncwarp();
    if (share) cl.sync();
    else __syncthreads();
}

// (G alpha)_i, alpha in shared memory: the sums of g_alpha
template <typename L, int CW>
__device__ __forceinline__ void lam_g_alpha(const LamArgs<L> &a, const L *al, int i, L (&out)[CW]) {
    const int h = a.g_w / 2;
    L sp[CW], sm[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) sp[c] = sm[c] = L(0);
    for (int e = 0; e < h; ++e) {
        const int cp = a.g_col[(size_t)e * a.nl + i], cm = a.g_col[(size_t)(h + e) * a.nl + i];
        const L vp = a.g_val[(size_t)e * a.nl + i], vm = a.g_val[(size_t)(h + e) * a.nl + i];
        if (cp >= 0)
#pragma unroll
            for (int c = 0; c < CW; ++c) sp[c] += vp * al[cp * CW + c];
        if (cm >= 0)
#pragma unroll
            for (int c = 0; c < CW; ++c) sm[c] += vm * al[cm * CW + c];
    }
#pragma unroll
    for (int c = 0; c < CW; ++c) out[c] = sp[c] - sm[c];
}

// the group's columns of U dof u of y_U (zeros past R)
template <typename L, int CW>
__device__ __forceinline__ Pack<L, CW> lam_load_y(const LamArgs<L> &a, int u, int c0, bool vec) {
    Pack<L, CW> o;
    const L *p = a.yU + (size_t)u * a.R + c0;
    if (vec) return *reinterpret_cast<const Pack<L, CW> *>(p);
#pragma unroll
    for (int c = 0; c < CW; ++c) o.v[c] = c0 + c < a.R ? p[c] : L(0);
    return o;
}

// sum of val(k, i) load(idx(k, i)) over the entries k of ELL row i (n rows, w entries, -1 past the
// row's end), in order; four entries' loads in flight
template <typename L, int CW, typename F>
__device__ __forceinline__ void lam_ell_gather(const int32_t *idx, const L *val, int w, int n, int i, L (&v)[CW],
                                               F &&load) {
#pragma unroll
    for (int c = 0; c < CW; ++c) v[c] = L(0);
    for (int k0 = 0; k0 < w; k0 += 4) {
        int id[4];
        L m[4];
        Pack<L, CW> t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) id[k] = k0 + k < w ? __ldg(idx + (size_t)(k0 + k) * n + i) : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (id[k] >= 0) {
                m[k] = __ldg(val + (size_t)(k0 + k) * n + i);
                t[k] = load(id[k]);
            }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (id[k] >= 0)
#pragma unroll
                for (int c = 0; c < CW; ++c) v[c] += m[k] * t[k].v[c];
    }
}

// the apply input entries of U dof u for the group's columns: FP32 paired, FP64 columns (the last
// dof of a subdomain zeroes the padding of its columns)
template <typename L, int CW>
__device__ __forceinline__ void lam_store_x(const LamArgs<L> &a, int u, int c0, const L (&v)[CW]) {
    const int4 t = a.u2x[u];
    if constexpr (std::is_same<L, float>::value) {
        const int R2 = (a.R + 1) / 2 * 2;
        L *p = a.x + (size_t)t.x * R2 + (size_t)(c0 >> 1) * t.y + t.z;
        if constexpr (CW == 1) p[c0 & 1] = v[0];
        else
#pragma unroll
            for (int c = 0; c < CW; c += 2)
                if (c0 + c < a.R) *reinterpret_cast<float2 *>(p + (size_t)(c >> 1) * t.y) = make_float2(v[c], v[c + 1]);
    } else {
        L *p = a.x + (size_t)t.x * a.R + (size_t)c0 * t.y;
#pragma unroll
        for (int c = 0; c < CW; ++c)
            if (c0 + c < a.R) {
                p[(size_t)c * t.y + t.z] = v[c];
                if (t.z == t.w - 1)
                    for (int k = t.w; k < t.y; ++k) p[(size_t)c * t.y + k] = L(0);
            }
    }
}
template <typename L, int CW>
__device__ __forceinline__ void lam_store_x16(const LamArgs<L> &a, const int4 *u2c, int u, int c0, const L (&v)[CW]) {
    const int4 t = u2c[u];
    __half *p = a.x16 + (size_t)t.x * a.R + (size_t)c0 * t.y;
#pragma unroll
    for (int c = 0; c < CW; ++c)
        if (c0 + c < a.R) {
            p[(size_t)c * t.y + t.z] = to_half(v[c]);
            if (t.z == t.w - 1)
                for (int k = t.w; k < t.y; ++k) p[(size_t)c * t.y + k] = __float2half(0.0f);
        }
}

// Grid: LC x groups CTAs in clusters of LC.  COND: sets the condition of the WHILE loop (continue
// while a right-hand side is active and fewer than limit iterations have run).  s.loops counts the
// iterations (zero before the first, which has no previous step to finish).
template <typename L, int CW, int COND>
__global__ void __launch_bounds__(LAM_THREADS, 1) k_lam_a(LamArgs<L> a, const int4 *u2c) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ LamShared<L, CW> sh;
    extern __shared__ __align__(16) unsigned char lam_dyn[];
    using P = Pack<L, CW>;
    const int grp = blockIdx.x / LC, rank = (int)cl.block_rank(), c0 = grp * CW;
    const bool first = *a.s.loops == 0;
    const L *sbeta = beta_of<L>(a.s);
    bool act[CW], any = false;
    L beta[CW], eta[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        const bool in = c0 + c < a.R;
        act[c] = in && a.s.active[c0 + c] != 0;
        any |= act[c];
        beta[c] = in ? sbeta[c0 + c] : L(0);
        eta[c] = L(0);
    }
    int n_act = 0;
    if (any) {          // (uniform over the cluster: it alone changes its columns' state, after this point)
        cluster_started_arrive();
        const int nl = a.nl, i0 = rank * LAM_THREADS + threadIdx.x;
        const size_t gb = (size_t)grp * nl;
        P *r = reinterpret_cast<P *>(a.r) + gb, *w = reinterpret_cast<P *>(a.w) + gb, *y = reinterpret_cast<P *>(a.y) + gb,
          *pv = reinterpret_cast<P *>(a.pv) + gb, *q = reinterpret_cast<P *>(a.q) + gb,
          *lam = reinterpret_cast<P *>(a.lam) + gb;
        const bool vec = CW > 1 && a.R % CW == 0;
        if (threadIdx.x < CW && c0 + threadIdx.x < a.R) sh.it[threadIdx.x] = a.s.iters[c0 + threadIdx.x];
        L s[CW], e[CW];
        if (!first) {
            // q = B y_U, (p_new, q), eta
#pragma unroll
            for (int c = 0; c < CW; ++c) s[c] = e[c] = L(0);
#pragma unroll 2
            for (int i = i0; i < nl; i += LC * LAM_THREADS) {
                const P yp = lam_load_y<L, CW>(a, a.bpm[i], c0, vec), ym = lam_load_y<L, CW>(a, a.bpm[nl + i], c0, vec);
                const P po = pv[i], yo = y[i];
                P qo;
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    qo.v[c] = yp.v[c] - ym.v[c];
                    two_add(s[c], e[c], p_next(po.v[c], yo.v[c], beta[c], act[c]) * qo.v[c], L(0));
                }
                q[i] = qo;
            }
            cluster_started_wait();
            cluster_sum<L, CW>(sh, 0, s, e, [&](int c, double pq) {
                const bool ac = c0 + c < a.R && a.s.active[c0 + c] != 0;
                const double yw = ac ? a.s.yw[c0 + c] : 0.0;
                const double et = (ac && pq != 0.0) ? yw / pq : 0.0;
                sh.step[c] = (L)et;
                if (ac) {
                    sh.it[c] += 1;
                    if (rank == 0) {
                        a.s.eta[c0 + c] = et;
                        a.s.yw_old[c0 + c] = yw;
                        a.s.iters[c0 + c] = sh.it[c];
                    }
                }
            });
#pragma unroll
            for (int c = 0; c < CW; ++c) eta[c] = sh.step[c];
        } else {
            cluster_started_wait();
        }
        // alpha from G^T r_new
        L *al = nullptr;
        if (a.nco > 0)
            cluster_alpha<L, CW>(a, lam_dyn, al, [&](int row) {
                P v = ld_cg(r + row);
                if (!first) {
                    const P qo = ld_cg(q + row);
#pragma unroll
                    for (int c = 0; c < CW; ++c) v.v[c] = r_next(v.v[c], qo.v[c], eta[c]);
                }
                return v;
            });
        // the step's updates, w = P r, (w, w) (every read of r by another CTA lies before
        // cluster_alpha's barrier)
#pragma unroll
        for (int c = 0; c < CW; ++c) s[c] = e[c] = L(0);
#pragma unroll 2
        for (int i = i0; i < nl; i += LC * LAM_THREADS) {
            P ro = r[i], wo;
            if (first) {
                P zero;
#pragma unroll
                for (int c = 0; c < CW; ++c) zero.v[c] = L(0);
                pv[i] = zero;
            } else {
                P po = pv[i], lo = lam[i];
                const P yo = y[i], qo = q[i];
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    po.v[c] = p_next(po.v[c], yo.v[c], beta[c], act[c]);
                    lo.v[c] = fma_l(eta[c], po.v[c], lo.v[c]);
                    ro.v[c] = r_next(ro.v[c], qo.v[c], eta[c]);
                }
                pv[i] = po;
                lam[i] = lo;
                r[i] = ro;
            }
            L ga[CW];
            if (al) lam_g_alpha<L, CW>(a, al, i, ga);
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                L xv = ro.v[c];
                if (al) xv += -ga[c];
                wo.v[c] = xv;
                two_add(s[c], e[c], xv * xv, L(0));
            }
            w[i] = wo;
        }
        cluster_sum<L, CW>(sh, 1, s, e, [&](int c, double ww) {
            // stop test; the columns' state to global memory from rank 0 (read by the other CTAs
            // before this reduction's barrier only, but for their own copy below)
            const double nw = sqrt(ww);
            const double xs = (nw > 0.0 && nw < INFINITY) ? ldexp(1.0, max(-126, min(126, -ilogb(nw)))) : 1.0;
            int on = 0;
            if (act_of(act, c)) {
                const double ref = a.s.nPd[c0 + c];
                on = !(nw <= a.tol * ref || sh.it[c] >= a.max_it);
                if (rank == 0) {
                    a.s.relres[c0 + c] = ref > 0 ? nw / ref : 0.0;
                    a.s.active[c0 + c] = on;
                }
            }
            if (rank == 0 && c0 + c < a.R) {
                a.s.xscale[c0 + c] = xs;
                a.s.xscale_f[c0 + c] = (float)xs;
            }
            sh.on[c] = on;
            sh.xsl[c] = (L)xs;
        });
#pragma unroll
        for (int c = 0; c < CW; ++c) n_act += sh.on[c];
        // x = B_D^T w
        if (n_act > 0) {
            const int nu = a.nu;
#pragma unroll 2
            for (int u = i0; u < nu; u += LC * LAM_THREADS) {
                L v[CW];
                lam_ell_gather<L, CW>(a.bdt_row, a.bdt_val, a.bdt_w, nu, u, v, [&](int row) { return ld_cg(w + row); });
                if (a.x16) {
#pragma unroll
                    for (int c = 0; c < CW; ++c) v[c] *= sh.xsl[c];
                    lam_store_x16<L, CW>(a, u2c, u, c0, v);
                } else {
                    lam_store_x<L, CW>(a, u, c0, v);
                }
            }
        }
    }
    // the groups' active columns: the last group to arrive publishes the total
    if (rank == 0 && threadIdx.x == 0) {
        const unsigned ng = gridDim.x / LC, add = (1u << 16) + (unsigned)n_act;
        const unsigned old = atomicAdd(a.s.counter, add);
        if ((old >> 16) == ng - 1) {
            const int total = (int)((old + add) & 0xffffu);
            *a.s.n_active = total;
            *a.s.counter = 0u;
            const int l = *a.s.loops + 1;
            *a.s.loops = l;
            if (COND) cudaGraphSetConditional(a.cond, (total > 0 && l < a.limit) ? 1u : 0u);
        }
    }
}

template <typename L, int CW>
__global__ void __launch_bounds__(LAM_THREADS, 1) k_lam_b(LamArgs<L> a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ LamShared<L, CW> sh;
    extern __shared__ __align__(16) unsigned char lam_dyn[];
    using P = Pack<L, CW>;
    const int grp = blockIdx.x / LC, rank = (int)cl.block_rank(), c0 = grp * CW;
    bool act[CW], any = false;
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        act[c] = c0 + c < a.R && a.s.active[c0 + c] != 0;
        any |= act[c];
    }
    if (!any) return;                      // every step of inactive columns is masked; uniform over the cluster
    const int nl = a.nl, i0 = rank * LAM_THREADS + threadIdx.x;
    const size_t gb = (size_t)grp * nl;
    P *w = reinterpret_cast<P *>(a.w) + gb, *z = reinterpret_cast<P *>(a.z) + gb, *y = reinterpret_cast<P *>(a.y) + gb,
      *pv = reinterpret_cast<P *>(a.pv) + gb;
    const bool vec = CW > 1 && a.R % CW == 0;
    // z = B_D y_U
#pragma unroll 2
    for (int i = i0; i < nl; i += LC * LAM_THREADS) {
        P zo;
        lam_ell_gather<L, CW>(a.bd_col, a.bd_val, a.bd_w, nl, i, zo.v,
                              [&](int u) { return lam_load_y<L, CW>(a, u, c0, vec); });
        z[i] = zo;
    }
    __syncwarp();
    cl.sync();                             // z is complete, and every CTA has started
    L *al = nullptr;
    if (a.nco > 0) {
        cluster_alpha<L, CW>(a, lam_dyn, al, [&](int row) { return ld_cg(z + row); });
    }
    // y = P z, (y, w)
    L s[CW], e[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) s[c] = e[c] = L(0);
#pragma unroll 2
    for (int i = i0; i < nl; i += LC * LAM_THREADS) {
        P yo = z[i];
        const P wo = w[i];
        L ga[CW];
        if (al) lam_g_alpha<L, CW>(a, al, i, ga);
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            if (al) yo.v[c] += -ga[c];
            two_add(s[c], e[c], yo.v[c] * wo.v[c], L(0));
        }
        y[i] = yo;
    }
    cluster_sum<L, CW>(sh, 0, s, e, [&](int c, double yw) {
        L be = L(0);
        if (c0 + c < a.R) {
            const double yo = a.s.yw_old[c0 + c];
            const double b = (a.s.iters[c0 + c] == 0 || yo == 0.0) ? 0.0 : yw / yo;
            be = (L)b;
            if (rank == 0) {
                a.s.yw[c0 + c] = yw;
                a.s.beta[c0 + c] = b;
                a.s.beta_f[c0 + c] = (float)b;
            }
        }
        sh.step[c] = be;
    });
    L beta[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) beta[c] = sh.step[c];
    // x = B^T p_new
    const int nu = a.nu;
#pragma unroll 4
    for (int u = i0; u < nu; u += LC * LAM_THREADS) {
        L v[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) v[c] = L(0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int sr = a.bt[(size_t)k * nu + u];
            if (sr != 0) {
                const int row = (sr > 0 ? sr : -sr) - 1;
                const P po = ld_cg(pv + row), yo = ld_cg(y + row);
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    const L pn = p_next(po.v[c], yo.v[c], beta[c], act[c]);
                    v[c] += sr > 0 ? pn : -pn;
                }
            }
        }
        lam_store_x<L, CW>(a, u, c0, v);
    }
}

// entry (i, c) of an interleaved FP64 vector pair <-> the grouped layout in L: r and lambda at the
// start of the iterations (columns past R zero), and back at their end.  n = groups nl CW entries.
template <typename L>
__global__ void k_group_enter(const double *r, const double *lam, L *rg, L *lg, int64_t nl, int R, int cw, int64_t n) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t gi = t / cw, g = gi / nl, i = gi % nl;
        const int c = (int)(g * cw + t % cw);
        rg[t] = c < R ? (L)r[i * R + c] : L(0);
        lg[t] = c < R ? (L)lam[i * R + c] : L(0);
    }
}
template <typename L>
__global__ void k_group_exit(const L *lg, const L *rg, double *lam, double *r, int64_t nl, int R, int cw) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nl * R; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / R;
        const int c = (int)(t % R);
        const int64_t o = ((int64_t)(c / cw) * nl + i) * cw + c % cw;
        lam[t] = (double)lg[o];
        r[t] = (double)rg[o];
    }
}
