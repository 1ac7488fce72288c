// Interface apply for wide blocks of right-hand sides (16 per streamed pass): the pipeline of
// k_apply_tma without a producer warp.
//
// With 16 right-hand sides the FP32 products bound the apply as much as the stream does: per 512
// operator entries a warp with 4 rows needs 128 packed FMAs and 20 16-byte shared loads (16 of x, 4 of
// the operator), and the loads alone take 80 clocks of the SM's shared memory.  Eight rows per warp
// halve the x loads (96 clocks per 1024 entries, 128 of the FMA pipes), but hold 128 accumulators and
// 32 operator entries per lane: about 190 registers, which two CTAs of four such warps have (255 each)
// and two CTAs of four and a producer warp do not (170).  So the copies are issued by the consumers: the last
// of the four warps to finish a stage refills it for the stage NS further on.  Two CTAs per SM, each
// with its own items, keep the SM busy across refills.
// Same items, tiles, per-lane order of operations and reduction as k_apply_tma: bitwise the same y.
// Measured (S_k^+, two CTAs per SM): peridynamic workload (346 MB, 16 right-hand sides) 92.8 -> 79.7 us,
// fractional workload (186 MB, 64 right-hand sides in four blocks) 169 -> 147 us; FP16 copy there 154 -> 141.
//
// Waits are bounded as in k_apply_tma; a wait that runs out sets *err, the warps stop at their next
// wait, and thread 0 waits (bounded) for the copies issued before the CTA returns.
#pragma once

constexpr int SELF_THREADS = 128;
constexpr int SELF_WARPS = SELF_THREADS / 32;
constexpr int SELF_RPW = 8;                         // rows per warp: 32 rows per item

template <int RC, int NS, typename MT>
__global__ void __launch_bounds__(SELF_THREADS, 2)
    k_apply_self(const CUtensorMap *maps, const CUtensorMap *xmaps, int use_sp, const SubdomainDesc *sd,
                 const int32_t *sched_ptr, const int32_t *sched_items, double *y, int R, const int *gate, int *err,
                 double oscale, long long wait_tries, int withhold, float *yf) {
    constexpr int CW = APPLY_CB / 4;                // columns per stage
    constexpr int MROW = CW * (int)sizeof(MT);
    constexpr int STAGE = apply_stage_bytes(RC, MROW, true);
    extern __shared__ __align__(128) unsigned char ring_raw[];
    unsigned char *ring = ring_raw + ((1024u - (smem_u32(ring_raw) & 1023u)) & 1023u);
    __shared__ uint64_t full[NS];
    __shared__ int done[NS], issued;                // warps finished with a stage; stages issued so far
    __shared__ volatile int abort_flag;
    if (gate && *gate == 0) return;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&full[s], 1);
            done[s] = 0;
        }
        issued = 0;
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int it0 = sched_ptr[blockIdx.x], it1 = sched_ptr[blockIdx.x + 1];
    const uint64_t stream_policy = l2_evict_first_policy();
    // the next stage to issue: item, first right-hand side, first column (every warp keeps the same)
    int pit = it0, pc0 = 0, pl0 = 0;
    ApplyItem pcur{}, pnxt{};
    if (it0 < it1) pcur = load_apply_item<ROWS_APPLY>(sched_items, sd, it0);
    if (it0 + 1 < it1) pnxt = load_apply_item<ROWS_APPLY>(sched_items, sd, it0 + 1);
    auto issue = [&](int q) {                       // one lane
        unsigned char *stg = ring + (q % NS) * STAGE;
        mbar_arrive_expect_tx(&full[q % NS], STAGE);
        tile_g2s_hint(stg, maps + 2 * pcur.k + use_sp, pl0, pcur.i0, &full[q % NS], stream_policy);
        tile_g2s(stg + 32 * MROW, xmaps + pcur.k, pl0, pc0 / 2, &full[q % NS]);
        atomicMax(&issued, q + 1);
    };
    auto advance = [&]() {
        pl0 += CW;
        if (pl0 < pcur.ncp) return;
        pl0 = 0;
        pc0 += RC;
        if (pc0 < R) return;
        pc0 = 0;
        ++pit;
        pcur = pnxt;
        if (pit + 1 < it1) pnxt = load_apply_item<ROWS_APPLY>(sched_items, sd, pit + 1);
    };
    for (int q = 0; q < NS; ++q) {
        if (pit >= it1) break;
        // withhold (fault injection for tests of the bounded waits): no copy is ever issued
        if (threadIdx.x == 0 && !withhold) issue(q);
        advance();
    }
    int q = 0;
    bool ok = true;
    ApplyItem nxt{};
    if (it0 < it1) nxt = load_apply_item<ROWS_APPLY>(sched_items, sd, it0);
    for (int it = it0; it < it1 && ok; ++it) {
        const ApplyItem cur = nxt;
        if (it + 1 < it1) nxt = load_apply_item<ROWS_APPLY>(sched_items, sd, it + 1);
        const int n = cur.n, ncp = cur.ncp, ib = cur.i0 + warp * SELF_RPW;
        for (int c0 = 0; c0 < R && ok; c0 += RC) {
            const int rc = min(RC, R - c0);
            float2 acc[SELF_RPW][RC / 2];
#pragma unroll
            for (int r = 0; r < SELF_RPW; ++r)
#pragma unroll
                for (int c = 0; c < RC / 2; ++c) acc[r][c] = make_float2(0.f, 0.f);
            for (int l0 = 0; l0 < ncp; l0 += CW, ++q) {
                const int s = q % NS;
                if (__any_sync(0xffffffffu, !mbar_wait(&full[s], (q / NS) & 1, wait_tries, &abort_flag) || abort_flag)) {
                    if (lane == 0) { atomicExch(err, 1); abort_flag = 1; }
                    ok = false;
                    break;
                }
                const MT *st = reinterpret_cast<const MT *>(ring + s * STAGE);
                const float *xs = reinterpret_cast<const float *>(ring + s * STAGE + 32 * MROW);
                if (ib < n) {
#pragma unroll
                    for (int j = 0; j < CW / 128; ++j)
                        rows_step_paired<RC, SELF_RPW, MT>(st + (warp * SELF_RPW) * CW + lane * 4 + j * 128, CW,
                                                           xs + j * 256 + lane * 4, acc);
                }
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    if (atomicAdd(&done[s], 1) == SELF_WARPS - 1) {
                        done[s] = 0;
                        __threadfence_block();
                        if (pit < it1 && !withhold) issue(q + NS);
                    }
                }
                if (pit < it1) advance();
            }
            if (!ok) break;
            // lane sums: groups of 4 rows and 8 columns, the shuffle tree of k_apply_tma
#pragma unroll
            for (int rh = 0; rh < SELF_RPW; rh += 4)
#pragma unroll
                for (int g0 = 0; g0 < RC; g0 += 8) {
                    float v[32];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            const float2 a2 = acc[rh + r][(g0 + c) / 2];
                            v[r * 8 + c] = (c & 1) ? a2.y : a2.x;
                        }
                    const float tot = warp_reduce_scatter<float, 32>(v, lane);
                    const int r = lane / 8, c = g0 + lane % 8, i = ib + rh + r;
                    if (c < rc && i < n) {
                        if (yf) yf[(cur.yoff + i) * R + c0 + c] = tot * (float)oscale;
                        else y[(cur.yoff + i) * R + c0 + c] = (double)tot * oscale;
                    }
                }
        }
    }
    __syncthreads();
    if (abort_flag && threadIdx.x == 0)             // let the copies already issued land
        for (int t = max(0, issued - NS); t < issued; ++t) mbar_wait(&full[t % NS], (t / NS) & 1);
}
