// Lambda-space work of a PCG iteration as one kernel per step, for more Lambda rows than the
// cluster kernels take (lambda_cluster.cuh).  Vectors hold the R right-hand sides interleaved (entry i of
// column c at i R + c); a lane takes V consecutive columns of a row (V = 4 or 2 where R is a multiple
// of it: one 16- or 8-byte access), and B, B_D, their transposes and G = B Z are read in ELL form.
// These kernels are bound by latency and by the load units; with one column per lane and 64-bit CSR
// indices the stop-test kernel of the fractional workload (30975 rows x 64) took 54 us.  Measured, the
// eight kernels of an iteration together: fractional 218 -> 108 us, peridynamic (38150 rows x 16)
// 90 -> 69 us, 82775 rows x 1 72 -> 63 us.
//
// Reductions: the rows are cut into tiles of RT = 8; block b owns the contiguous tiles
// [b tpb, (b + 1) tpb) (tpb from n and the grid only).  A (tile, chunk of columns) unit takes four lanes
// per column group: lane h adds rows h and h + 4, and the four are added as ((h0 + h2) + (h1 + h3)),
// in L.  The block adds its tile sums per column, 32 tiles at a time: four threads per column take 8 tiles
// each in order and keep running sums, added as ((0 + 1) + (2 + 3)) at the end; the last block to arrive
// adds the blocks' partials (32 lanes per column, then the lane tree).  FP32 sums are kept as compensated
// pairs (TwoSum) from the tile sums on: FP64 additions cost a warp 64 clocks each on this GPU (the pairs
// differ from FP64 sums by 2^-46 of the sum of magnitudes, where the FP32 products and tile sums err by
// 2^-30, 2^-24 at most: errors against exact sums 1.0000003 of those with FP64 tile sums on average, 1.00003 at
// most, 16 k to 83 k rows), and for the same reason the scalars are updated by one thread per column (one lane of a warp each, 64 columns
// took about 20 us of that kernel).  R, V and the number of warps only decide who adds what
// when, never the order, so a column's sums do not depend on its batch.
#pragma once

constexpr int RT = 8;
constexpr int TILE_THREADS = 1024;      // threads of a tile-reduction block (one block per SM)
constexpr int TILE_COLS = 64;           // columns per pass
constexpr int TILE_ROUND = 32;          // tiles per round

// one 1024-thread CTA per SM: the warps of four 256-thread CTAs, a quarter of the partials for
// the last block to add
constexpr int TILE_MAX_BLOCKS = 152;
inline int tile_blocks(int64_t n) {
    const int64_t nt = (n + RT - 1) / RT;
    return (int)std::max<int64_t>(1, std::min<int64_t>(TILE_MAX_BLOCKS, (nt + 1) / 2));
}

// V consecutive columns at p (aligned to V entries where V > 1)
template <int V, typename L> __device__ __forceinline__ Pack<L, V> ld_pack(const L *p) {
    return *reinterpret_cast<const Pack<L, V> *>(p);
}
template <int V, typename L> __device__ __forceinline__ void st_pack(L *p, const Pack<L, V> &v) {
    *reinterpret_cast<Pack<L, V> *>(p) = v;
}

// a sum as stored per block: FP64, or a compensated FP32 pair
template <typename L> struct PartialOf { using type = double; };
template <> struct PartialOf<float> { using type = float2; };
__device__ __forceinline__ double make_partial(double s, double) { return s; }
__device__ __forceinline__ float2 make_partial(float s, float e) { return make_float2(s, e); }
__device__ __forceinline__ void add_partial(double &s, double &, double p) { s += p; }
__device__ __forceinline__ void add_partial(float &s, float &e, float2 p) { two_add(s, e, p.x, p.y); }
__device__ __forceinline__ double ld_partial(const double *p) { return __ldcg(p); }
__device__ __forceinline__ float2 ld_partial(const float2 *p) { return __ldcg(p); }

// f(i, c0): the addends of row i, columns c0 .. c0 + V - 1, called once each (i < n)
template <int V, typename L, typename F>
__device__ __forceinline__ void tile_reduce(int64_t n, int R, typename PartialOf<L>::type *partial, F &&f) {
    __shared__ L ts[TILE_ROUND * (TILE_COLS + 1)];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int64_t ntiles = (n + RT - 1) / RT;
    const int64_t tpb = (ntiles + gridDim.x - 1) / gridDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * tpb, t1 = min(ntiles, t0 + tpb);
    for (int cc0 = 0; cc0 < R; cc0 += TILE_COLS) {
        const int ncol = min(TILE_COLS, R - cc0), ng = (ncol + V - 1) / V;
        const int cw = ng >= 5 ? 8 : (ng >= 3 ? 4 : (ng == 2 ? 2 : 1));
        const int ulanes = 4 * cw, upw = 32 / ulanes, nchunk = (ng + cw - 1) / cw;
        const int ju = lane / ulanes, jl = lane % ulanes, h = jl / cw, cj = jl % cw;
        const int col = threadIdx.x >> 2, quarter = threadIdx.x & 3;
        L as = L(0), ae = L(0);
        for (int64_t tb = t0; tb < t1; tb += TILE_ROUND) {
            const int ntl = (int)min((int64_t)TILE_ROUND, t1 - tb), units = ntl * nchunk;
            for (int ub = warp * upw; ub < units; ub += (TILE_THREADS / 32) * upw) {
                const int u = ub + ju, tl = u / nchunk, g = (u % nchunk) * cw + cj;
                const bool ok = u < units && g < ng;
                Pack<L, V> v;
#pragma unroll
                for (int k = 0; k < V; ++k) v.v[k] = L(0);
                if (ok) {
                    const int64_t i0 = (tb + tl) * RT + h;
                    Pack<L, V> a = v, b = v;
                    if (i0 < n) a = f(i0, cc0 + g * V);
                    if (i0 + 4 < n) b = f(i0 + 4, cc0 + g * V);
#pragma unroll
                    for (int k = 0; k < V; ++k) v.v[k] = a.v[k] + b.v[k];
                }
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    v.v[k] += __shfl_down_sync(0xffffffffu, v.v[k], 2 * cw);
                    v.v[k] += __shfl_down_sync(0xffffffffu, v.v[k], cw);
                    if (ok && h == 0) ts[tl * (TILE_COLS + 1) + g * V + k] = v.v[k];
                }
            }
            __syncthreads();
            if (threadIdx.x < 4 * ncol)
                for (int t = 8 * quarter; t < min(ntl, 8 * quarter + 8); ++t)
                    two_add(as, ae, ts[t * (TILE_COLS + 1) + col], L(0));
            __syncthreads();
        }
        // the four quarters (whole warps take part: lanes past the columns add zeros)
        if (warp < (4 * ncol + 31) / 32) {
#pragma unroll
            for (int o = 1; o <= 2; o *= 2) {
                const L bs = __shfl_down_sync(0xffffffffu, as, o), be = __shfl_down_sync(0xffffffffu, ae, o);
                two_add(as, ae, bs, be);
            }
            if (quarter == 0 && col < ncol)
                partial[(int64_t)(cc0 + col) * gridDim.x + blockIdx.x] = make_partial(as, ae);
        }
    }
}

// last block: column totals over the nb row-block partials (fixed order) and the PCG scalar update, one
// thread per column:
//   NPD:   ||P d|| and the initial state;      CHECK: ||w|| and the active mask;
//   BETA:  (y,w) and beta = (y,w)/(y,w)_old;    ETA:   (p,q) and eta = (y,w)/(p,q).
template <int MODE, typename L>
__device__ void finish_scalars(const typename PartialOf<L>::type *partial, int nb, int R, PcgScalars s, double tol,
                               int max_it) {
    using P = typename PartialOf<L>::type;
    __shared__ int n_act;
    __shared__ double tot[TILE_COLS];
    constexpr int FIN_GROUP = 5;            // partials per lane loaded together
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) n_act = 0;
    for (int cc0 = 0; cc0 < R; cc0 += TILE_COLS) {
        const int ncol = min(TILE_COLS, R - cc0);
        __syncthreads();
        for (int cl = warp; cl < ncol; cl += TILE_THREADS / 32) {
            const P *pc = partial + (int64_t)(cc0 + cl) * nb;
            L v = L(0), ve = L(0);
            for (int b0 = lane; b0 < nb; b0 += 32 * FIN_GROUP) {
                P pv[FIN_GROUP];
#pragma unroll
                for (int m = 0; m < FIN_GROUP; ++m)
                    if (b0 + 32 * m < nb) pv[m] = ld_partial(pc + b0 + 32 * m);
#pragma unroll
                for (int m = 0; m < FIN_GROUP; ++m)
                    if (b0 + 32 * m < nb) add_partial(v, ve, pv[m]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const L bs = __shfl_down_sync(0xffffffffu, v, o), be = __shfl_down_sync(0xffffffffu, ve, o);
                two_add(v, ve, bs, be);
            }
            if (lane == 0) tot[cl] = std::is_same<L, float>::value ? (double)v + (double)ve : (double)v;
        }
        __syncthreads();
        if (threadIdx.x < ncol) {
            const int c = cc0 + threadIdx.x;
            const double v = tot[threadIdx.x];
            if (MODE == FIN_NPD) {
                s.nPd[c] = sqrt(v);
                s.active[c] = 1;
                s.iters[c] = 0;
                s.yw_old[c] = 1.0;
                s.relres[c] = 1.0;
                s.eta[c] = 0.0;
                s.beta[c] = 0.0;
                s.eta_f[c] = 0.0f;
                s.beta_f[c] = 0.0f;
                s.xscale_f[c] = 1.0f;
            } else if (MODE == FIN_CHECK) {
                const double nw = sqrt(v), ref = s.nPd[c];
                // a power of two that FP32 holds too (the FP32 pass scales with the same factor)
                const double xs = (nw > 0.0 && nw < INFINITY) ? ldexp(1.0, max(-126, min(126, -ilogb(nw)))) : 1.0;
                s.xscale[c] = xs;
                s.xscale_f[c] = (float)xs;
                int act = s.active[c];
                if (act) s.relres[c] = ref > 0 ? nw / ref : 0.0;
                if (act && (nw <= tol * ref || s.iters[c] >= max_it)) act = 0;
                s.active[c] = act;
                if (act) atomicAdd(&n_act, 1);
            } else if (MODE == FIN_BETA) {
                s.yw[c] = v;
                const double b = (s.iters[c] == 0 || s.yw_old[c] == 0.0) ? 0.0 : v / s.yw_old[c];
                s.beta[c] = b;
                s.beta_f[c] = (float)b;
            } else {
                const bool act = s.active[c] != 0;
                const double e = (act && v != 0.0) ? s.yw[c] / v : 0.0;
                s.eta[c] = e;
                s.eta_f[c] = (float)e;
                if (act) { s.yw_old[c] = s.yw[c]; s.iters[c] += 1; }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (MODE == FIN_NPD) *s.n_active = R;
        if (MODE == FIN_CHECK) *s.n_active = n_act;
        *s.counter = 0u;
    }
}

// (a, b) per column with the scalar update of MODE (grid tile_blocks(n))
template <int MODE>
__global__ void __launch_bounds__(TILE_THREADS) k_dot_final(const double *__restrict__ a, const double *__restrict__ b,
                                                            int64_t n, int R, double *partial, PcgScalars s, double tol,
                                                            int max_it) {
    tile_reduce<1, double>(n, R, partial, [&](int64_t i, int c) { return Pack<double, 1>{{a[i * R + c] * b[i * R + c]}}; });
    if (arrive_last(s.counter)) finish_scalars<MODE, double>(partial, gridDim.x, R, s, tol, max_it);
}

// (G alpha)_i of V columns (the order of the sums of g_alpha)
template <int V, typename L>
__device__ __forceinline__ Pack<L, V> g_alpha_v(const LamArgs<L> &a, const L *alpha, int64_t i, int c0) {
    const int h = a.g_w / 2;
    Pack<L, V> sp, sm;
#pragma unroll
    for (int k = 0; k < V; ++k) sp.v[k] = sm.v[k] = L(0);
    for (int e = 0; e < h; ++e) {
        const int cp = a.g_col[(size_t)e * a.nl + i], cm = a.g_col[(size_t)(h + e) * a.nl + i];
        const L vp = a.g_val[(size_t)e * a.nl + i], vm = a.g_val[(size_t)(h + e) * a.nl + i];
        if (cp >= 0) {
            const Pack<L, V> t = ld_pack<V>(alpha + (size_t)cp * a.R + c0);
#pragma unroll
            for (int k = 0; k < V; ++k) sp.v[k] += vp * t.v[k];
        }
        if (cm >= 0) {
            const Pack<L, V> t = ld_pack<V>(alpha + (size_t)cm * a.R + c0);
#pragma unroll
            for (int k = 0; k < V; ++k) sm.v[k] += vm * t.v[k];
        }
    }
#pragma unroll
    for (int k = 0; k < V; ++k) sp.v[k] -= sm.v[k];
    return sp;
}

// Start of a PCG iteration (after the coarse kernel formed alpha from G^T r_new): the previous
// iteration's updates p = p_new, lambda += eta p, r = r_new, then w = P r = r - G alpha,
// (w, w) and the stop test.  The active flags read here are those p_new was formed with: the
// last block changes them only after every block has arrived.  COND: the last block also
// counts the iteration and sets the condition of the WHILE loop (continue while a
// right-hand side is active and fewer than limit iterations have run, so the loop ends
// whatever the scalars hold); a separate instantiation, as profilers skip kernels that set
// graph conditions.  (alpha: NULL without a coarse space)
template <int COND, typename L, int V>
__global__ void __launch_bounds__(TILE_THREADS) k_check_update(LamArgs<L> a, const L *alpha,
                                                               typename PartialOf<L>::type *partial) {
    const L *eta = eta_of<L>(a.s), *beta = beta_of<L>(a.s);
    const int R = a.R;
    tile_reduce<V, L>(a.nl, R, partial, [&](int64_t i, int c) {
        const int64_t t = i * R + c;
        const Pack<L, V> e = ld_pack<V>(eta + c), be = ld_pack<V>(beta + c), po = ld_pack<V>(a.pv + t),
                         yo = ld_pack<V>(a.y + t), ro = ld_pack<V>(a.r + t), qo = ld_pack<V>(a.q + t);
        const Pack<int, V> act = ld_pack<V>(a.s.active + c);
        Pack<L, V> lo = ld_pack<V>(a.lam + t), pn, x, o;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            pn.v[k] = p_next(po.v[k], yo.v[k], be.v[k], act.v[k] != 0);
            lo.v[k] = fma_l(e.v[k], pn.v[k], lo.v[k]);
            x.v[k] = r_next(ro.v[k], qo.v[k], e.v[k]);
        }
        st_pack<V>(a.pv + t, pn);
        st_pack<V>(a.lam + t, lo);
        st_pack<V>(a.r + t, x);
        if (alpha) {
            const Pack<L, V> ga = g_alpha_v<V>(a, alpha, i, c);
#pragma unroll
            for (int k = 0; k < V; ++k) x.v[k] += -ga.v[k];
        }
        st_pack<V>(a.w + t, x);
#pragma unroll
        for (int k = 0; k < V; ++k) o.v[k] = x.v[k] * x.v[k];
        return o;
    });
    if (arrive_last(a.s.counter)) {
        finish_scalars<FIN_CHECK, L>(partial, gridDim.x, R, a.s, a.tol, a.max_it);
        if (COND && threadIdx.x == 0) {
            const int l = *a.s.loops + 1;
            *a.s.loops = l;
            cudaGraphSetConditional(a.cond, (*a.s.n_active > 0 && l < a.limit) ? 1u : 0u);
        }
    }
}

// y = P z = z - G alpha with (y, w) and the BETA update.  Grid tile_blocks(nl).
template <typename L, int V>
__global__ void __launch_bounds__(TILE_THREADS) k_project_dot(LamArgs<L> a, const L *alpha,
                                                              typename PartialOf<L>::type *partial) {
    const int R = a.R;
    tile_reduce<V, L>(a.nl, R, partial, [&](int64_t i, int c) {
        const int64_t t = i * R + c;
        Pack<L, V> x = ld_pack<V>(a.z + t), o;
        const Pack<L, V> wo = ld_pack<V>(a.w + t);
        if (alpha) {
            const Pack<L, V> ga = g_alpha_v<V>(a, alpha, i, c);
#pragma unroll
            for (int k = 0; k < V; ++k) x.v[k] += -ga.v[k];
        }
        st_pack<V>(a.y + t, x);
#pragma unroll
        for (int k = 0; k < V; ++k) o.v[k] = x.v[k] * wo.v[k];
        return o;
    });
    if (arrive_last(a.s.counter)) finish_scalars<FIN_BETA, L>(partial, gridDim.x, R, a.s, 0.0, 0);
}

// q = B y_U with (p_new, q) and the ETA update (p_new formed per row, stored by the next
// iteration's k_check_update).  Grid tile_blocks(nl).
template <typename L, int V>
__global__ void __launch_bounds__(TILE_THREADS) k_gather_b_eta(LamArgs<L> a, typename PartialOf<L>::type *partial) {
    const L *beta = beta_of<L>(a.s);
    const int R = a.R;
    tile_reduce<V, L>(a.nl, R, partial, [&](int64_t i, int c) {
        const int64_t t = i * R + c;
        const Pack<L, V> yp = ld_pack<V>(a.yU + (size_t)a.bpm[i] * R + c), ym = ld_pack<V>(a.yU + (size_t)a.bpm[a.nl + i] * R + c),
                         po = ld_pack<V>(a.pv + t), yo = ld_pack<V>(a.y + t), be = ld_pack<V>(beta + c);
        const Pack<int, V> act = ld_pack<V>(a.s.active + c);
        Pack<L, V> x, o;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            x.v[k] = yp.v[k] - ym.v[k];
            o.v[k] = p_next(po.v[k], yo.v[k], be.v[k], act.v[k] != 0) * x.v[k];
        }
        st_pack<V>(a.q + t, x);
        return o;
    });
    if (arrive_last(a.s.counter)) finish_scalars<FIN_ETA, L>(partial, gridDim.x, R, a.s, 0.0, 0);
}

// z = B_D y_U; one thread per (row, column group), groups fastest
template <typename L, int V> __global__ void __launch_bounds__(256) k_gather_bd_v(LamArgs<L> a) {
    const unsigned ng = (unsigned)a.R / V, n = (unsigned)a.nl;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (uint64_t)n * ng; t += (uint64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / ng), c = (int)(t % ng) * V;
        Pack<L, V> v;
        lam_ell_gather<L, V>(a.bd_col, a.bd_val, a.bd_w, (int)n, i, v.v,
                             [&](int u) { return ld_pack<V>(a.yU + (size_t)u * a.R + c); });
        st_pack<V>(a.z + (size_t)i * a.R + c, v);
    }
}

// the apply inputs x = B_D^T w (FP16 input of the tensor-core apply where a.x16) and x = B^T p_new; one
// thread per (U dof, column group), groups fastest: R consecutive entries read per Lambda row, and
// eight neighbouring dofs' entries written side by side
template <typename L, int V>
__global__ void __launch_bounds__(256) k_gather_w_v(LamArgs<L> a, const int4 *u2c, const int *gate) {
    if (*gate == 0) return;
    const L *xs = xscale_of<L>(a.s);
    const unsigned ng = (unsigned)a.R / V, n = (unsigned)a.nu;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (uint64_t)n * ng; t += (uint64_t)gridDim.x * blockDim.x) {
        const int u = (int)(t / ng), c = (int)(t % ng) * V;
        L v[V];
        lam_ell_gather<L, V>(a.bdt_row, a.bdt_val, a.bdt_w, (int)n, u, v,
                             [&](int row) { return ld_pack<V>(a.w + (size_t)row * a.R + c); });
        if (a.x16) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] *= xs[c + k];
            lam_store_x16<L, V>(a, u2c, u, c, v);
        } else {
            lam_store_x<L, V>(a, u, c, v);
        }
    }
}
template <typename L, int V> __global__ void __launch_bounds__(256) k_gather_p_v(LamArgs<L> a, const int *gate) {
    if (*gate == 0) return;
    const L *beta = beta_of<L>(a.s);
    const unsigned ng = (unsigned)a.R / V, n = (unsigned)a.nu;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (uint64_t)n * ng; t += (uint64_t)gridDim.x * blockDim.x) {
        const int u = (int)(t / ng), c = (int)(t % ng) * V;
        const Pack<L, V> be = ld_pack<V>(beta + c);
        const Pack<int, V> act = ld_pack<V>(a.s.active + c);
        int sr[2];
        Pack<L, V> po[2], yo[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) sr[k] = a.bt[(size_t)k * n + u];
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (sr[k] != 0) {
                const size_t o = (size_t)((sr[k] > 0 ? sr[k] : -sr[k]) - 1) * a.R + c;
                po[k] = ld_pack<V>(a.pv + o);
                yo[k] = ld_pack<V>(a.y + o);
            }
        L v[V];
#pragma unroll
        for (int j = 0; j < V; ++j) v[j] = L(0);
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (sr[k] != 0)
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const L pn = p_next(po[k].v[j], yo[k].v[j], be.v[j], act.v[j] != 0);
                    v[j] += sr[k] > 0 ? pn : -pn;
                }
        lam_store_x<L, V>(a, u, c, v);
    }
}

// alpha = (G^T G)^-1 G^T v inside the iterations, v = z (RNEW 0) or r_new = r - eta q (RNEW 1); grid
// (floating subdomains, psplit slices of the entry range, column groups).  Block (f, j, g) sums
// slice j into gpart (a thread's entries in ascending order, PGU in flight; warps in order).  Small
// coarse spaces (fused 1): the last block to arrive adds the slices and applies (G^T G)^-1 in FP64.
// FP32 beyond that (fused 2, one slice): the last of a column group's blocks to arrive applies the FP32
// copy of (G^T G)^-1, stored transposed, thread i summing over j in ascending order.  FP64 beyond
// that: k_coarse_solve follows.
constexpr int PGU = 8;
template <int RNEW, typename L, int V>
__global__ void __launch_bounds__(256) k_proj_v(LamArgs<L> a, double *gpart, double *gsum, L *alpha, int psplit, int fused) {
    extern __shared__ double gs_dyn[];
    __shared__ L red[8][3][V];
    const int f = blockIdx.x, c = blockIdx.z * V, R = a.R, nco = a.nco;
    const int64_t e0 = a.gt_range[4 * f], e1 = a.gt_range[4 * f + 1];
    const int co_off = a.gt_co[2 * f], nq = a.gt_co[2 * f + 1];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int64_t chunk = (e1 - e0 + psplit - 1) / psplit, l0 = e0 + blockIdx.y * chunk, l1 = min(e1, l0 + chunk);
    Pack<L, V> eta;
    if (RNEW) eta = ld_pack<V>(eta_of<L>(a.s) + c);
    const L *vec = RNEW ? a.r : a.z;
    L acc[3][V];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int k = 0; k < V; ++k) acc[q][k] = L(0);
    constexpr int U = V >= 4 ? PGU / 2 : PGU;
    for (int64_t b = l0 + threadIdx.x; b < l1; b += U * (int64_t)blockDim.x) {
        int row[U];
        Pack<L, V> x[U];
#pragma unroll
        for (int m = 0; m < U; ++m) row[m] = b + m * (int64_t)blockDim.x < l1 ? a.gt_row[b + m * (int64_t)blockDim.x] : -1;
#pragma unroll
        for (int m = 0; m < U; ++m)
            if (row[m] >= 0) {
                x[m] = ld_pack<V>(vec + (size_t)row[m] * R + c);
                if (RNEW) {
                    const Pack<L, V> qo = ld_pack<V>(a.q + (size_t)row[m] * R + c);
#pragma unroll
                    for (int k = 0; k < V; ++k) x[m].v[k] = r_next(x[m].v[k], qo.v[k], eta.v[k]);
                }
            }
#pragma unroll
        for (int m = 0; m < U; ++m)
            if (row[m] >= 0) {
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q < nq) {
                        const L w = a.gt_w[q * a.gt_n + b + m * (int64_t)blockDim.x];
#pragma unroll
                        for (int k = 0; k < V; ++k) acc[q][k] += w * x[m].v[k];
                    }
            }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (q < nq)
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const L t = warp_sum(acc[q][k]);
                if (lane == 0) red[warp][q][k] = t;
            }
    __syncthreads();
    if (threadIdx.x < nq * V) {
        const int q = threadIdx.x / V, k = threadIdx.x % V;
        L x = 0;
        for (int ww = 0; ww < 8; ++ww) x += red[ww][q][k];
        gpart[((int64_t)(co_off + q) * psplit + blockIdx.y) * R + c + k] = (double)x;
    }
    if (!fused) return;
    if constexpr (std::is_same<L, float>::value) {
        if (fused == 2) {
            if (!arrive_last_col(a.s.colcnt, blockIdx.z)) return;
            float *gc = reinterpret_cast<float *>(gs_dyn);       // n_co x V entries of G^T v
            for (int t = threadIdx.x; t < nco * V; t += blockDim.x) {
                const int j = t / V, k = t % V;
                double g = 0;
                for (int s = 0; s < psplit; ++s) g += __ldcg(gpart + ((int64_t)j * psplit + s) * R + c + k);
                gc[t] = (float)g;
            }
            __syncthreads();
            for (int i = threadIdx.x; i < nco; i += blockDim.x) {
                // j ascending; the loads of 16 consecutive j in flight together
                Pack<float, V> o;
#pragma unroll
                for (int k = 0; k < V; ++k) o.v[k] = 0.0f;
                int j = 0;
                for (; j + 16 <= nco; j += 16) {
                    float gv[16];
#pragma unroll
                    for (int m = 0; m < 16; ++m) gv[m] = __ldg(a.ginv32 + (size_t)(j + m) * nco + i);
#pragma unroll
                    for (int m = 0; m < 16; ++m)
#pragma unroll
                        for (int k = 0; k < V; ++k) o.v[k] = __fmaf_rn(gv[m], gc[(j + m) * V + k], o.v[k]);
                }
                for (; j < nco; ++j) {
                    const float gv = __ldg(a.ginv32 + (size_t)j * nco + i);
#pragma unroll
                    for (int k = 0; k < V; ++k) o.v[k] = __fmaf_rn(gv, gc[j * V + k], o.v[k]);
                }
                st_pack<V>(alpha + (size_t)i * R + c, o);
            }
            if (threadIdx.x == 0) a.s.colcnt[blockIdx.z] = 0u;
            return;
        }
    }
    if (!arrive_last(a.s.counter)) return;
    double *gs = gsum ? gsum : gs_dyn;
    for (int t = threadIdx.x; t < nco * R; t += blockDim.x) {
        const int i = t / R, cc = t % R;
        double g = 0;
        for (int j = 0; j < psplit; ++j) g += __ldcg(gpart + ((int64_t)i * psplit + j) * R + cc);
        gs[t] = g;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nco * R; t += blockDim.x) {
        const int i = t / R, cc = t % R;
        double v = 0;
        for (int j = 0; j < nco; ++j) v += a.ginv[(int64_t)i * nco + j] * gs[(int64_t)j * R + cc];
        alpha[t] = (L)v;
    }
    if (threadIdx.x == 0) *a.s.counter = 0u;
}
