// sic_kernels.cu -- sm_103a kernel of the SIC step.
//
// k_step runs one whole step (or one of its halves) in a single launch, over
// one or many simulations:
//   1. a block works on one simulation at a time; each of its warps claims
//      runs of work items (up to 32 R consecutive tracers of one sheet, R per
//      lane) from that simulation's cursor, gathers E at each tracer (linear
//      weighting between the two nodes), kicks, drifts, and writes the tracer
//      to the other state buffer;
//   2. it deposits the segment from each of its tracers to the next one
//      (Sec. 2.3, Eq. overlap and Eq. rho_sum) into the block's shared-memory
//      copy of the simulation's int64 charge mesh.  The tracer after the
//      warp's last one is read from the input buffer and pushed again by the
//      warp itself, so warps and blocks never wait for one another;
//   3. when the simulation has no unclaimed items left, the block adds its
//      mesh into the global mesh with int64 atomics and counts its items on
//      the simulation's ticket; the block that completes the count runs the
//      epilogue: the exact integer field solve, the field energy, the
//      diagnostic row, and the buffer swap.  The block then moves to the
//      simulation with the most unclaimed items, until none has any.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sic_item.cuh"

namespace sic {

namespace {

// Field solve of one simulation (Sec. 2.1 with C = 1) by the block holding
// its last ticket: sm (nx u64) and sE (nx floats) are this block's scratch.
//   P_j = sum_{i<j} mesh_i, D_j = nx P_j - j Q (= nx sigma E'_j exactly),
//   K_j = nx D_j - sum_j D_j (= nx^2 sigma E_j, zero mean), all integers,
//   with sum_j D_j = nx (nx - 1) Q / 2 - nx sum_i i mesh_i (from
//   sum_j P_j = sum_i (nx - 1 - i) mesh_i), so it needs no pass of its own;
//   kick table Ek_j = K_j e_scale rounded once to FP32, field energy from
//   the squares of K_j 2^-60 summed in FP32 within a warp and FP64 across.
// Everything it reads from global memory (the mesh, the step's sums, the
// scalars) is requested at once, so it waits for memory once.
// The double-precision field and density for the host are recomputed from
// mesh_last on request (k_field_out), so this path has no FP64 per cell.
__device__ void field_epilogue(const SimDev &S, int record, unsigned long long *sm, float *sE, Shared &sh)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = S.nx;
    if (tid >= 32 && tid < 41) {
        const unsigned long long *src = tid < 36 ? &S.acc->ke[tid - 32] : tid < 40 ? &S.acc->p[tid - 36] : &S.acc->maxseg;
        sh.pre[tid - 32] = __ldcg(src);
    } else if (tid == 64) {
        sh.pre_step = __ldcg(&S.sc->step);
    } else if (tid == 65) {
        sh.pre_we = __ldcg(&S.sc->we);
    } else if (tid == 66) {
        sh.pre_err = __ldcg(&S.sc->err);
    } else if (tid == 67) {
        sh.pre_hold = __ldcg(&S.sc->hold);
    } else if (tid == 68) {
        sh.pre_wk = __ldcg(&S.sc->wk);
    }
    for (int j = tid; j < nx; j += 4 * B) {
        unsigned long long mv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            mv[k] = j + k * B < nx ? __ldcg(S.mesh + j + k * B) : 0ull;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (j + k * B < nx) {
                sm[j + k * B] = mv[k];
                S.mesh[j + k * B] = 0ull;
                S.mesh_last[j + k * B] = (long long)mv[k];
            }
        }
    }
    __syncthreads();
    const int per = (nx + B - 1) / B;
    const int j0 = min(tid * per, nx), j1 = min(j0 + per, nx);
    long long lsum = 0;
    __int128 m1 = 0;  // sum_j j mesh_j over this thread's cells
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        const long long mv = (long long)sm[j];
        lsum += mv;
        m1 += (__int128)j * mv;
    }
    long long incl = lsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        m1 += shfl_down_i128(m1, o);
    if (lane == 31)
        sh.w64[warp] = incl;
    if (lane == 0) {
        sh.hi[warp] = (long long)(m1 >> 64);
        sh.lo[warp] = (long long)(unsigned long long)m1;
    }
    __syncthreads();
    long long before = 0, qtot = 0;
    __int128 M1 = 0;
    for (int w = 0; w < NW; ++w) {
        if (w < warp)
            before += sh.w64[w];
        qtot += sh.w64[w];
        M1 += make_i128(sh.hi[w], sh.lo[w]);
    }
    const long long run0 = incl - lsum + before;
    const __int128 sumD = (__int128)((long long)nx * (nx - 1) / 2) * qtot - (__int128)nx * M1;

    // K from cell to cell: D_{j+1} = D_j + nx mesh_j - Q
    float wloc = 0.f;
    const int mode_k = S.mode_k;
    float mre = 0.f, mim = 0.f;  // this thread's part of sum_j K_j 2^-60 exp(-2 pi i j k / nx)
    __int128 D = (__int128)nx * run0 - (__int128)j0 * qtot;
    __int128 K = (__int128)nx * D - sumD;
    if (S.deposit == SIC_DEPOSIT_FIRST) {
        // charge on the nodes: the trapezoid rule between nodes makes the node
        // field the mean of K at j and j + 1 (K_nx = K_0), 2 E_j = K_j + K_{j+1}
#pragma unroll 1
        for (int j = j0; j < j1; ++j) {
            D += (__int128)nx * (long long)sm[j] - qtot;
            const __int128 Kn = (__int128)nx * D - sumD;
            const Norm128 n2 = norm128(K + Kn);
            sE[j] = __fmul_rn(norm_to_float(n2, S.ek_exp - 1), S.ek_mant);
            const float kn = norm_to_float(n2, -61);
            wloc = __fmaf_rn(kn, kn, wloc);
            if (mode_k)
                mode_add(kn, j, mode_k, nx, mre, mim);
            K = Kn;
        }
    } else {
#pragma unroll 2
        for (int j = j0; j < j1; ++j) {
            const Norm128 nk = norm128(K);
            sE[j] = __fmul_rn(norm_to_float(nk, S.ek_exp), S.ek_mant);
            const float kn = norm_to_float(nk, -60);
            wloc = __fmaf_rn(kn, kn, wloc);
            if (mode_k)
                mode_add(kn, j, mode_k, nx, mre, mim);
            D += (__int128)nx * (long long)sm[j] - qtot;
            K = (__int128)nx * D - sumD;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        wloc = __fadd_rn(wloc, __shfl_down_sync(0xffffffffu, wloc, o));
    if (lane == 0)
        sh.da[warp] = (double)wloc;
    if (mode_k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mre = __fadd_rn(mre, __shfl_down_sync(0xffffffffu, mre, o));
            mim = __fadd_rn(mim, __shfl_down_sync(0xffffffffu, mim, o));
        }
        if (lane == 0) {
            sh.mre[warp] = mre;
            sh.mim[warp] = mim;
        }
    }
    __syncthreads();
    for (int j = tid; j < nx; j += B) {
        const int j1n = (j + 1 == nx) ? 0 : j + 1;
        S.Ek[j] = make_float2(sE[j], sE[j1n] - sE[j]);
    }
    // the scalars: four threads, each one chain of (slow) FP64 arithmetic
    SimScalars *sc = S.sc;
    const long long step = sh.pre_step;
    double *row = nullptr;
    long long slot = 0;
    if (record && (tid == 0 || tid == 32 || tid == 64 || tid == 128)) {
        slot = step % S.hist_len;
        row = S.hist + 4 * slot;
    }
    auto limbs = [](const unsigned long long *l) -> double {
        const unsigned __int128 u = (unsigned __int128)l[0] + ((unsigned __int128)l[1] << 32) +
                                    ((unsigned __int128)l[2] << 64) + ((unsigned __int128)l[3] << 96);
        return i128_words_to_double((unsigned long long)u, (unsigned long long)(u >> 64));
    };
    if (tid == 32 && record)
        row[1] = S.ke_scale * times_pow2(limbs(sh.pre), -S.ke_u);
    if (tid == 64 && record)
        row[2] = S.p_scale * times_pow2(limbs(sh.pre + 4), -S.p_u);
    if (tid == 96) {
        double w = 0.0;
        for (int i = 0; i < NW; ++i)
            w += sh.da[i];
        sc->we = w * S.we_scale;
    }
    if (tid == 128 && mode_k) {
        // W_k = dx / nx |E^_k|^2 (half at k = nx/2) = (2 or 1) / nx we_scale |Z|^2
        double re = 0.0, im = 0.0;
        for (int i = 0; i < NW; ++i) {
            re += (double)sh.mre[i];
            im += (double)sh.mim[i];
        }
        if (record)
            S.mhist[slot] = sh.pre_wk;
        sc->wk = (2 * mode_k == nx ? 1.0 : 2.0) / nx * S.we_scale * (re * re + im * im);
    }
    if (tid == 0) {
        SimAccum *ac = S.acc;
        const long long mm = (long long)sh.pre[8];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            ac->ke[k] = ac->p[k] = 0ull;
        ac->maxseg = 0ull;
        if (record) {
            row[0] = sh.pre_we;
            row[3] = (double)qtot;
            sc->step = step + 1;
        }
        sc->q_total = qtot;
        sc->maxseg = mm;
        unsigned err = sh.pre_err, hold = sh.pre_hold;
        if (S.strict && mm > ((long long)nx << 16))
            err |= SIC_ERR_SEGLONG;
        // the position format holds a segment exactly while it is shorter than
        // 2 box lengths; one of 1.5 or more ends the run with a range error.
        // Each end moves less than half a box per step, so a segment cannot
        // get from below 1.5 box lengths to 2.5 or more (where its difference
        // would alias to less than 1.5) in one step unseen
        if (mm >= ((long long)(3 * nx) << 15))
            err |= SIC_ERR_RANGE;
        // hold the simulation (its later steps leave it as it is) when it
        // needs the host: an error, or a particle longer than the refinement
        // length (Sec. 2.6), to be split before the run goes on.  The decision
        // is the simulation's own, so it stops at the same step alone or in
        // any batch
        if (err)
            hold |= SIC_HOLD_ERROR;
        if (S.refine_seg > 0 && mm > S.refine_seg)
            hold |= SIC_HOLD_REFINE;
        if (err != sh.pre_err)
            sc->err = err;
        if (hold != sh.pre_hold)
            sc->hold = hold;
    }
}

template <bool PUSH, bool DEPOSIT, bool PER_Q, bool STAGED, bool GEN>
__global__ void __launch_bounds__(B, SIC_K1_MIN_BLOCKS) k_step(const LaunchArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Shared &sh = *reinterpret_cast<Shared *>(smem);
    const int nx_max = A.nx_max;
    unsigned long long *mesh_region = reinterpret_cast<unsigned long long *>(smem + kSharedHead);
    Hist hist;
    hist.lo = reinterpret_cast<unsigned *>(mesh_region);
    hist.hi = hist.lo + nx_max;
    Hist diff;  // the difference array of long particles: nx_max + 2 cells
    diff.lo = reinterpret_cast<unsigned *>(mesh_region + nx_max);
    diff.hi = diff.lo + nx_max + 2;
    float2 *ek = reinterpret_cast<float2 *>(mesh_region + nx_max + nx_max + 2);
    char *stage_base = reinterpret_cast<char *>(smem) + stage_offset(nx_max);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float ks = A.kick_scale;
    const int drift = (PUSH && DEPOSIT) ? 1 : A.drift;  // a full step always drifts
    char *my_stage = stage_base + (size_t)warp * WarpBuf<PER_Q, STAGED>::bytes;
    unsigned short *tasks =
        reinterpret_cast<unsigned short *>(stage_base + (size_t)NW * WarpBuf<PER_Q, STAGED>::bytes) + warp * WT;
    unsigned phase = 0;      // bit s: parity of stage s's next completion
    int s = 0;               // the stage the warp's next item lands in
    bool timed_out = false;
    if (STAGED) {
        if (tid < 2 * NW)
            mbar_init(&sh.mbar[tid >> 1][tid & 1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }

    // the first simulation: the one that holds this block's proportional
    // share of the launch's items
    int cur;
    {
        const long long target = ((2ll * blockIdx.x + 1) * (long long)A.n_items) / (2ll * gridDim.x);
        int lo = 0, hi = A.n_slots - 1;  // last slot with slot_begin <= target
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (A.slot_begin[mid] <= target)
                lo = mid;
            else
                hi = mid - 1;
        }
        cur = lo;
    }
    unsigned rerr = 0, mseg = 0;
    unsigned mlen = 0;  // longest crossing box particle, position units
    long long ake = 0, ap = 0;  // this lane's KE and P sums (units 2^-ke_u, 2^-p_u)
    bool first = true;          // the block's first simulation of the launch
    bool triggered = false;     // the next launch in the stream may start
    unsigned seen = 0;          // lane 0: the simulation's claim cursor as last seen
    unsigned done_old = 0;      // thread 0: blocks counted out before this one
    bool done_early = false;

    while (cur >= 0) {
        // ---- enter simulation cur: its descriptor into shared memory (the
        // launch's table does not change while it runs)
        for (int i = tid; i < (int)(sizeof(SimDev) / 4); i += B)
            reinterpret_cast<unsigned *>(&sh.sim)[i] = reinterpret_cast<const unsigned *>(A.sims + cur)[i];
        __syncthreads();
        const SimDev &S = sh.sim;
        const WorkItem *items = S.items;
        const int n_s = A.slot_begin[cur + 1] - A.slot_begin[cur];
        const int nx = S.nx;
        if (DEPOSIT) {
            for (int j = tid; j < nx; j += B) {
                hist.lo[j] = 0u;
                hist.hi[j] = 0u;
            }
            for (int j = tid; j < nx + 2; j += B) {
                diff.lo[j] = 0u;
                diff.hi[j] = 0u;
            }
        }
        if (tid == 0) {
            sh.diff_used = 0;
            sh.taken = 0;
            sh.ke[0] = sh.ke[1] = sh.p[0] = sh.p[1] = 0ull;
        }
        if (first) {
            // a launch that may start before the previous one in its stream
            // has finished waits here: everything below may be its output
            griddep_wait();
            first = false;
        }
        // one round trip: the hold and buffer words, the kick table and each
        // warp's first claim
        if (tid == 0) {
            sh.hold = *(volatile unsigned *)&S.sc->hold;
            sh.buf = *(volatile unsigned *)&S.sc->buf;
        }
        if (PUSH) {
            for (int j = tid; j < nx; j += B)
                ek[j] = S.Ek[j];
        }

        // ---- each warp claims runs of consecutive items (guided: a claim is
        // the fraction claim_q of what it saw left, at least claim_min items)
        // and streams them through its two stages.  A run's claim is made
        // when the run before the previous one ends, so its result has had a
        // whole run to arrive when it is needed.  With staging, an item's
        // descriptor is copied into shared memory while the item before it is
        // pushed, and its data copies start halfway through that item.
        unsigned *cursor = A.cursor + cur;
        const float q = A.claim_q;
        const int claim_min = max(1, A.claim_min);
        unsigned c_old = 0, c_want = 0;  // lane 0: the claim in flight
        auto claim_issue = [&]() {
            if (lane == 0) {
                const int left = n_s - (int)min(seen, (unsigned)n_s);
                c_want = left > 0 ? (unsigned)max(claim_min, (int)((float)left * q)) : 0u;
                c_old = c_want ? atomicAdd(cursor, c_want) : (unsigned)n_s;
            }
        };
        auto claim_take = [&](int &a, int &n) {  // the first use of the claim's result
            if (lane == 0)
                seen = c_old + c_want;
            const unsigned o = __shfl_sync(0xffffffffu, c_old, 0);
            const unsigned w = __shfl_sync(0xffffffffu, c_want, 0);
            a = (int)o;
            n = (int)o < n_s ? min((int)w, n_s - (int)o) : 0;
        };
        claim_issue();  // before the hold is known: a held simulation drops it
        __syncthreads();

        // a full step leaves a held simulation (set by an earlier launch's
        // epilogue, so the same for every block of this one) as it is: its
        // items are all marked claimed, so no block picks it again in this
        // launch.  An explicit deposit or push still runs.
        if (PUSH && DEPOSIT && sh.hold) {
            if (tid == 0)
                atomicAdd(cursor, (unsigned)n_s);
            __syncthreads();  // the block's own pick below sees it taken
        } else {
        const bool track_all = S.refine_seg > 0 && S.refine_seg < (1ll << 16);  // refinement below a cell
        const int src = (int)sh.buf;
        const unsigned *Uin = S.U[src];
        const float *Vin = S.V[src];
        unsigned *Uout = S.U[src ^ 1];
        float *Vout = S.V[src ^ 1];
        const int32_t *Qh = S.Qh;
        int a, n;
        claim_take(a, n);
        claim_issue();  // the next run's claim, in flight through this run
        int count = 0;
        if (STAGED) {
            if (n > 0 && !timed_out && lane == 0) {
                desc_fetch(&sh.desc[warp][s].w, items + a);
                desc_wait();
                stage_issue<PER_Q>(sh.desc[warp][s].w, Uin, Vin, Qh, my_stage + s * WarpBuf<PER_Q, true>::stage,
                                   &sh.mbar[warp][s]);
            }
            __syncwarp();
        }
        while (n > 0) {
            int na = 0, nn = 0;
            bool took = false;
            count += n;
            for (int i = a; i < a + n && !timed_out; ++i) {
                int nxt = i + 1;
                if (nxt == a + n) {
                    claim_take(na, nn);
                    claim_issue();  // the run after it, in flight through the next run
                    took = true;
                    nxt = nn > 0 ? na : -1;
                }
                if (!STAGED && lane == 0 && i + 2 < a + n) {
                    // lane 0 reads the next descriptor to start its copies:
                    // fetch the one after it into L1 now (both of its sectors),
                    // so that read does not wait on L2
                    const char *pf = reinterpret_cast<const char *>(items + i + 2);
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(pf));
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(pf + sizeof(WorkItem) - 1));
                }
                const WorkItem W = STAGED ? sh.desc[warp][s].w : items[i];
                const WorkItemPL *plw = (GEN && S.pl != nullptr) ? S.pl + i : nullptr;
                if (STAGED) {
                    // the next item's descriptor comes in while this one is
                    // pushed; its copies start halfway through this item
                    if (nxt >= 0 && lane == 0)
                        desc_fetch(&sh.desc[warp][s ^ 1].w, items + nxt);
                    const bool ok = mbar_wait_bounded(&sh.mbar[warp][s], (phase >> s) & 1u);
                    phase ^= 1u << s;
                    if (!__all_sync(0xffffffffu, ok)) {
                        // give up (the next item's copies have not started): only count items
                        timed_out = true;
                        mbar_drain(&sh.mbar[warp][s], ((phase >> s) & 1u) ^ 1u);
                        if (nxt >= 0 && lane == 0)
                            desc_wait();
                        break;
                    }
                    auto mid = [&]() {
                        if (nxt >= 0 && lane == 0) {
                            desc_wait();
                            stage_issue<PER_Q>(sh.desc[warp][s ^ 1].w, Uin, Vin, Qh,
                                               my_stage + (s ^ 1) * WarpBuf<PER_Q, true>::stage, &sh.mbar[warp][s ^ 1]);
                        }
                    };
                    char *st = my_stage + s * WarpBuf<PER_Q, true>::stage;
                    if (W.count == WT)
                        do_item<PUSH, DEPOSIT, PER_Q, true, true, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh,
                                                                  nx, ks, drift, rerr, st, st, tasks, ake, ap, mseg, mlen, plw,
                                                                  S.deposit, S.seg_q, track_all, mid);
                    else
                        do_item<PUSH, DEPOSIT, PER_Q, false, true, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh,
                                                                   nx, ks, drift, rerr, st, st, tasks, ake, ap, mseg, mlen, plw,
                                                                   S.deposit, S.seg_q, track_all, mid);
                    __syncwarp();
                    s ^= 1;
                } else {
                    auto mid = []() {};
                    if (W.count == WT)
                        do_item<PUSH, DEPOSIT, PER_Q, true, false, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh,
                                                                   nx, ks, drift, rerr, my_stage, my_stage, tasks, ake, ap, mseg, mlen,
                                                                   plw, S.deposit, S.seg_q, track_all, mid);
                    else
                        do_item<PUSH, DEPOSIT, PER_Q, false, false, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh,
                                                                    nx, ks, drift, rerr, my_stage, my_stage, tasks, ake, ap, mseg, mlen,
                                                                    plw, S.deposit, S.seg_q, track_all, mid);
                }
            }
            if (!took) {
                claim_take(na, nn);
                claim_issue();
            }
            a = na;
            n = nn;
        }
        if (lane == 0)
            atomicAdd(&sh.taken, count);
        if (!triggered) {
            // this block has no more items to start: the next launch in the
            // stream may begin (it waits for this one's end before it reads)
            griddep_launch_dependents();
            triggered = true;
        }

        // ---- leave: fold the block's mesh and sums into the simulation's,
        // take an item ticket, run the field epilogue if it completes it
        if (PUSH) {
            const Acc128 k2 = i64_warp_sum(ake);
            const Acc128 p2 = i64_warp_sum(ap);
            if (lane == 0) {
                sh.wke[warp][0] = (long long)k2.lo;
                sh.wke[warp][1] = k2.hi;
                sh.wp[warp][0] = (long long)p2.lo;
                sh.wp[warp][1] = p2.hi;
            }
            ake = 0;
            ap = 0;
        }
        if (DEPOSIT) {
            mseg = max(mseg, (unsigned)(((unsigned long long)mlen * (unsigned)(nx << SIC_POS_WIND_BITS)) >> 16));
            mlen = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                mseg = max(mseg, __shfl_down_sync(0xffffffffu, mseg, o));
            if (lane == 0)
                sh.wmseg[warp] = mseg;
            mseg = 0;
        }
        __syncthreads();
        if (DEPOSIT) {
            if (sh.diff_used)
                add_diff_prefix(hist, diff, nx, sh);
            for (int j = tid; j < nx; j += B) {
                const unsigned long long h = hist.get(j);
                if (h)
                    atomicAdd(S.mesh + j, h);
            }
        }
        if (rerr >> 30)  // a step of half a box or more, or a sum that is not finite
            atomicOr(&S.sc->err, SIC_ERR_RANGE);
        rerr = 0;
        if (STAGED && timed_out && lane == 0)
            atomicOr(&S.sc->err, SIC_ERR_TIMEOUT);
        if (tid == 0) {
            SimAccum *ac = S.acc;
            if (PUSH) {
                // the block's 128-bit sums, added limb by limb
                Acc128 k{sh.ke[0], (long long)sh.ke[1]}, pm{sh.p[0], (long long)sh.p[1]};
                for (int w = 0; w < NW; ++w) {
                    acc_add(k, Acc128{(unsigned long long)sh.wke[w][0], sh.wke[w][1]});
                    acc_add(pm, Acc128{(unsigned long long)sh.wp[w][0], sh.wp[w][1]});
                }
                const unsigned kl[4] = {(unsigned)k.lo, (unsigned)(k.lo >> 32), (unsigned)k.hi,
                                        (unsigned)((unsigned long long)k.hi >> 32)};
                const unsigned pl[4] = {(unsigned)pm.lo, (unsigned)(pm.lo >> 32), (unsigned)pm.hi,
                                        (unsigned)((unsigned long long)pm.hi >> 32)};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (kl[i])
                        atomicAdd(&ac->ke[i], (unsigned long long)kl[i]);
                    if (pl[i])
                        atomicAdd(&ac->p[i], (unsigned long long)pl[i]);
                }
            }
            if (DEPOSIT) {
                unsigned m = 0;
                for (int w = 0; w < NW; ++w)
                    m = max(m, sh.wmseg[w]);
                if (m)
                    atomicMax(&ac->maxseg, (unsigned long long)m);
            }
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            // only a block that took items counts them: a block whose claims
            // all came too late adds nothing, and must not read a completed
            // count as its own (that simulation's epilogue would run twice)
            const unsigned taken = (unsigned)sh.taken;
            sh.last = 0;
            if (taken) {
                const unsigned t = atomicAdd(A.tickets + cur, taken);
                sh.last = (t + taken == (unsigned)n_s) ? 1 : 0;
            }
            // a launch of one simulation: this block claims nothing more, so
            // it counts itself out now and reads the count after the epilogue
            if (A.n_slots == 1) {
                done_old = atomicAdd(A.done, 1u);
                done_early = true;
            }
        }
        __syncthreads();
        if (sh.last) {
            __threadfence();
            if (DEPOSIT)
                field_epilogue(S, A.record, mesh_region, reinterpret_cast<float *>(ek), sh);
            if (tid == 0) {
                if (PUSH)
                    S.sc->buf = (unsigned)(src ^ 1);
                if (!DEPOSIT) {  // the epilogue did not consume the sums: drop them
                    SimAccum *ac = S.acc;
                    for (int k = 0; k < 4; ++k)
                        ac->ke[k] = ac->p[k] = 0ull;
                    ac->maxseg = 0ull;
                }
                A.tickets[cur] = 0u;
            }
        }
        }  // not held

        // ---- next: the simulation with the most unclaimed items, if any
        // (a launch of one simulation has none)
        int most = 0;
        cur = -1;
        if (A.n_slots > 1) {
            int best = -1;
            for (int j = tid; j < A.n_slots; j += B) {
                const int left = (A.slot_begin[j + 1] - A.slot_begin[j]) - (int)*(volatile unsigned *)(A.cursor + j);
                if (left > most) {
                    most = left;
                    best = j;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int m2 = __shfl_down_sync(0xffffffffu, most, o);
                const int b2 = __shfl_down_sync(0xffffffffu, best, o);
                if (m2 > most) {
                    most = m2;
                    best = b2;
                }
            }
            if (lane == 0) {
                sh.pick_n[warp] = most;
                sh.pick_s[warp] = best;
            }
            __syncthreads();
            most = 0;
            for (int w = 0; w < NW; ++w)
                if (sh.pick_n[w] > most) {
                    most = sh.pick_n[w];
                    cur = sh.pick_s[w];
                }
            if (cur >= 0)  // its cursor as the search saw it
                seen = (unsigned)(A.slot_begin[cur + 1] - A.slot_begin[cur] - most);
        }
        __syncthreads();  // the picks and the epilogue's scratch are free again
    }

    // the last block out rewinds the claim cursors for the next launch
    if (tid == 0) {
        if (!done_early) {
            __threadfence();
            done_old = atomicAdd(A.done, 1u);
        }
        sh.last = (done_old + 1 == gridDim.x) ? 1 : 0;
    }
    __syncthreads();
    if (sh.last) {
        for (int j = tid; j < A.n_slots; j += B)
            A.cursor[j] = 0u;
        if (tid == 0)
            *A.done = 0u;
    }
}

template <bool P, bool D, bool Q, bool G, bool L>
cudaError_t prep(size_t smem)
{
    static size_t done = 0;
    if (smem > done) {
        cudaError_t e = cudaFuncSetAttribute(k_step<P, D, Q, G, L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess)
            return e;
        done = smem;
    }
    return cudaSuccess;
}

template <bool P, bool D, bool Q, bool G, bool L>
cudaError_t run(const LaunchArgs &a, int grid, cudaStream_t s)
{
    const size_t smem = step_smem_bytes(a.nx_max, G, Q);
    cudaError_t e = prep<P, D, Q, G, L>(smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(B);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e2 = cudaLaunchKernelEx(&cfg, k_step<P, D, Q, G, L>, a);
    count_launches(1);
    return e2 != cudaSuccess ? e2 : cudaGetLastError();
}

template <bool P, bool D, bool Q, bool G>
int occ(int nx_max)
{
    const size_t smem = step_smem_bytes(nx_max, G, Q);
    if (prep<P, D, Q, G, false>(smem) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step<P, D, Q, G, false>, B, smem) != cudaSuccess)
        return 0;
    return n;
}

// a.gen: some simulation of the launch deposits other than box particles;
// that variant handles every kind
template <bool P, bool D, bool G>
cudaError_t run_pd(const LaunchArgs &a, int grid, bool per_q, cudaStream_t s)
{
    if (a.gen)
        return per_q ? run<P, D, true, G, true>(a, grid, s) : run<P, D, false, G, true>(a, grid, s);
    return per_q ? run<P, D, true, G, false>(a, grid, s) : run<P, D, false, G, false>(a, grid, s);
}

template <bool P, bool D, bool G>
int occ_pd(int nx_max, bool per_q)
{
    return per_q ? occ<P, D, true, G>(nx_max) : occ<P, D, false, G>(nx_max);
}

// The double-precision node field E_j and density rho_j of the latest
// deposit, recomputed from its exact charge mesh (one block of 1024 threads).
// Fourier amplitudes |X^_k| = |sum_j X_j exp(-2 pi i j k / nx)| of the FP64
// density (field 0) or node field (field 1) that k_field_out wrote, one block
// per k = 0 .. nx/2, in a fixed order of additions (Sec. 3.2).
__global__ void __launch_bounds__(256) k_spectrum(const SimDev S, int field)
{
    __shared__ double s_re[8], s_im[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = S.nx, k = blockIdx.x;
    const double *X = field ? S.E64 : S.rho64;
    double re = 0.0, im = 0.0;
    for (int j = tid; j < nx; j += 256) {
        const int idx = (int)(((long long)j * k) % nx);
        double sn, cs;
        sincospi(2.0 * idx / nx, &sn, &cs);
        re = fma(X[j], cs, re);
        im = fma(-X[j], sn, im);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, o);
        im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        s_re[warp] = re;
        s_im[warp] = im;
    }
    __syncthreads();
    if (tid == 0) {
        re = 0.0;
        im = 0.0;
        for (int w = 0; w < 8; ++w) {
            re += s_re[w];
            im += s_im[w];
        }
        S.spec[k] = hypot(re, im);
    }
}

__global__ void __launch_bounds__(1024) k_field_out(const SimDev S)
{
    constexpr int BB = 1024, NWW = BB / 32;
    __shared__ long long s_w[NWW];
    __shared__ long long s_hi[NWW], s_lo[NWW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = S.nx;
    const int per = (nx + BB - 1) / BB;
    const int j0 = min(tid * per, nx), j1 = min(j0 + per, nx);
    long long lsum = 0;
    for (int j = j0; j < j1; ++j)
        lsum += S.mesh_last[j];
    long long incl = lsum;
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    if (lane == 31)
        s_w[warp] = incl;
    __syncthreads();
    long long before = 0, qtot = 0;
    for (int w = 0; w < NWW; ++w) {
        if (w < warp)
            before += s_w[w];
        qtot += s_w[w];
    }
    const long long run0 = incl - lsum + before;
    __int128 dsum = 0;
    long long run = run0;
    for (int j = j0; j < j1; ++j) {
        dsum += (__int128)nx * run - (__int128)j * qtot;
        run += S.mesh_last[j];
    }
    for (int o = 16; o > 0; o >>= 1)
        dsum += shfl_down_i128(dsum, o);
    if (lane == 0) {
        s_hi[warp] = (long long)(dsum >> 64);
        s_lo[warp] = (long long)(unsigned long long)dsum;
    }
    __syncthreads();
    __int128 sumD = 0;
    for (int w = 0; w < NWW; ++w)
        sumD += make_i128(s_hi[w], s_lo[w]);
    run = run0;
    const bool nodes = S.deposit == SIC_DEPOSIT_FIRST;  // E_j = (K_j + K_{j+1}) / 2
    for (int j = j0; j < j1; ++j) {
        const long long mj = S.mesh_last[j];
        const __int128 d = (__int128)nx * run - (__int128)j * qtot;
        const __int128 K = (__int128)nx * d - sumD;
        if (nodes) {
            const __int128 Kn = (__int128)nx * ((__int128)nx * (run + mj) - (__int128)(j + 1) * qtot) - sumD;
            S.E64[j] = i128_to_double(K + Kn) * (0.5 * S.E_scale);
        } else {
            S.E64[j] = i128_to_double(K) * S.E_scale;
        }
        S.rho64[j] = i128_to_double((__int128)nx * mj - qtot) * S.rho_scale;
        run += mj;
    }
}

__global__ void k_expand_horizontal(uint32_t *U, float *V, const uint32_t *ut, int32_t n, const float *vs,
                                    const int64_t *off, int32_t M)
{
    const long long total = (long long)M * n;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(g / n);
        const int i = (int)(g - (long long)s * n);
        U[off[s] + i] = ut[i];
        V[off[s] + i] = vs[s];
    }
}

}  // namespace

size_t step_smem_bytes(int nx_max, bool staged, bool per_q)
{
    // shared head, mesh lo/hi [nx], diff [nx + 2], E [nx + 1] (the epilogue
    // reuses mesh and E), then the warps' staging buffers
    // then per warp one staging buffer (two when staged) and a task list
    const size_t buf = staged ? (per_q ? WarpBuf<true, true>::bytes : WarpBuf<false, true>::bytes)
                              : (per_q ? WarpBuf<true, false>::bytes : WarpBuf<false, false>::bytes);
    return stage_offset(nx_max) + (size_t)NW * buf + (size_t)NW * WT * sizeof(unsigned short);
}

// Blocks of the step kernel that the SM's shared memory holds (registers cap
// them at SIC_K1_MIN_BLOCKS by the launch bounds).
static int blocks_by_smem(size_t smem)
{
    static int per_sm = 0;
    if (per_sm == 0) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess && v > 0)
            per_sm = v;
        else
            per_sm = 228 * 1024;
    }
    const int n = (int)((size_t)per_sm / (smem + 1024));  // 1 KB reserved per block
    return std::min(n, SIC_K1_MIN_BLOCKS);
}

// Stage items through shared memory unless the staging buffers would cost an
// SM a block (large meshes): occupancy hides more latency than staging.
bool step_staged(int nx_max, bool per_q)
{
    return blocks_by_smem(step_smem_bytes(nx_max, true, per_q)) >= blocks_by_smem(step_smem_bytes(nx_max, false, per_q));
}

static long long g_launches = 0;
void count_launches(int64_t n) { __atomic_add_fetch(&g_launches, n, __ATOMIC_RELAXED); }
int64_t launches() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

cudaError_t launch_step_kernel(const LaunchArgs &a, int grid, Mode mode, bool per_q, cudaStream_t s)
{
    switch (mode) {
    case MODE_STEP: {
        bool staged = step_staged(a.nx_max, per_q);
        if (a.staging == 1)
            staged = false;
        else if (a.staging == 2)
            staged = step_smem_bytes(a.nx_max, true, per_q) <= 227 * 1024;
        if (staged)
            return run_pd<true, true, true>(a, grid, per_q, s);
        return run_pd<true, true, false>(a, grid, per_q, s);
    }
    case MODE_DEPOSIT:
        return run_pd<false, true, false>(a, grid, per_q, s);
    default:
        return run_pd<true, false, false>(a, grid, per_q, s);
    }
}

int step_blocks_per_sm(int nx_max, Mode mode, bool per_q)
{
    switch (mode) {
    case MODE_STEP:
        if (step_staged(nx_max, per_q))
            return occ_pd<true, true, true>(nx_max, per_q);
        return occ_pd<true, true, false>(nx_max, per_q);
    case MODE_DEPOSIT:
        return occ_pd<false, true, false>(nx_max, per_q);
    default:
        return occ_pd<true, false, false>(nx_max, per_q);
    }
}

cudaError_t launch_field_out(const SimDev &sim, cudaStream_t s)
{
    k_field_out<<<1, 1024, 0, s>>>(sim);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_spectrum(const SimDev &sim, int field, cudaStream_t s)
{
    k_spectrum<<<sim.nx / 2 + 1, 256, 0, s>>>(sim, field);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_expand_horizontal(uint32_t *U, float *V, const uint32_t *u_template, int32_t n_template,
                                     const float *v_sheet, const int64_t *sheet_offset, int32_t n_sheets,
                                     cudaStream_t s)
{
    k_expand_horizontal<<<1216, 256, 0, s>>>(U, V, u_template, n_template, v_sheet, sheet_offset, n_sheets);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace sic

namespace sic {
namespace {

// ------------------------------------------------------------ moments ----
// Number density n and current density j of the box particles of the
// current state (Sec. 2.3, Eq. rho_sum and Eq. j_sum: zero order on cells;
// Sec. 2.4: first order on the nodes x_j = j dx, the velocity interpolated
// linearly along each particle).  FP64, atomics into n and j (physical units:
// n = charge / length, j = n v).
//
// One warp per work item, 8 consecutive tracers per lane: the loads are whole
// 128-byte lines, and a lane sums what its particles leave in one cell before
// it adds it to the mesh.  Cells and fractions come exactly from the 32.32
// cell coordinates.
//
// The FP64 pipe (two lanes a cycle and SM) bounds it, so a particle is cut
// into what its two end cells get, once per lane whatever its length, and the
// cells between, which all get the same and cost no arithmetic (first order:
// one addition a node), only their atomics; with kMomentCells of them or more
// they are shared out over the lanes.  Integers and FP32 numbers are turned
// into FP64 by their bits, and the reciprocal of the length is one
// third-order step from the FP32 one.  The diagnostics of 512 x 2048 folded
// tracers on 512 cells (both orders, a deposit, the field and two spectra) take
// 0.46 ms, of which the moments 88 and 186 us as calls; 0.72 ms with one mesh
// for all blocks, 1.59 ms with every cell's share worked out as well, 49.5 ms
// with one thread per work item.
constexpr int kMomentCells = 8;
// Two warps a block: items differ in cost by their cells, and small blocks leave
// a shorter tail (first order 211 us a call with eight warps)
constexpr int kMomentThreads = 64;

// v 2^-32 for v < 2^52, exactly: one FP64 subtraction instead of a conversion
__device__ __forceinline__ double cells_double(unsigned long long v)
{
    return __hiloint2double((int)(0x41300000u | (unsigned)(v >> 32)), (int)(unsigned)v) - 1048576.0;
}

// An FP32 number in FP64 by its bits (denormals: zero)
__device__ __forceinline__ double widen(float f)
{
    const unsigned w = __float_as_uint(f), e = w & 0x7f800000u;
    const unsigned hi = (w & 0x80000000u) | (((w & 0x7fffffffu) >> 3) + (e == 0x7f800000u ? 0x70000000u : 0x38000000u));
    return e == 0u ? 0.0 : __hiloint2double((int)hi, (int)(w << 29));
}

// 1 / x for x = len 2^-32 > 0: with e = 1 - x y, 1 / x = y (1 + e + e^2 + ...)
// to third order from the FP32 reciprocal y (e below 2^-21, so the rest is
// below 2^-63)
__device__ __forceinline__ double cells_recip(unsigned long long len, double x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(span_to_float((long long)len)));
    const double y0 = widen(__fmul_rn(y, 4294967296.0f));
    const double e = fma(-x, y0, 1.0);
    return fma(y0, fma(e, e, e), y0);
}

// What a lane's consecutive particles leave in one cell: the cell's own share
// (zero order), or its lower and upper node's (first order)
template <int W>
struct MomentRun {
    double *n, *j;
    int nx, cell;
    double sn[W + 1], sj[W + 1];
    __device__ __forceinline__ MomentRun(double *n_, double *j_, int nx_) : n(n_), j(j_), nx(nx_), cell(-1) {}
    __device__ __forceinline__ void flush()
    {
        if (cell >= 0) {
            atomicAdd(n + cell, sn[0]);
            atomicAdd(j + cell, sj[0]);
            if (W == 1) {
                const int c1 = cell + 1 == nx ? 0 : cell + 1;
                atomicAdd(n + c1, sn[W]);
                atomicAdd(j + c1, sj[W]);
            }
        }
    }
    __device__ __forceinline__ void add(int c, const double (&pn)[W + 1], const double (&pj)[W + 1])
    {
        if (c != cell) {
            flush();
            cell = c;
#pragma unroll
            for (int k = 0; k <= W; ++k) {
                sn[k] = pn[k];
                sj[k] = pj[k];
            }
        } else {
#pragma unroll
            for (int k = 0; k <= W; ++k) {
                sn[k] += pn[k];
                sj[k] += pj[k];
            }
        }
    }
};

// scratch: `copies` times a copy of n and one of j beside it (262 K tracers on 128
// cells: 74 and 79 us a call for the two orders with the copies in two arrays,
// 61 and 73 so); one copy: n and j themselves
template <int W>
__global__ void __launch_bounds__(kMomentThreads) k_moments(const SimDev S, double inv_dx, double unit_q, double unit_v, double *n,
                                                 double *j, double *scratch, int copies)
{
    const int nx = S.nx, nx4 = nx << SIC_POS_WIND_BITS;
    const int lane = threadIdx.x & 31;
    const int src = (int)S.sc->buf;
    const unsigned *U = S.U[src];
    const float *V = S.V[src];
    const int32_t *Qh = S.Qh;
    if (copies > 1) {
        n = scratch + (size_t)(blockIdx.x % copies) * 2 * nx;
        j = n + nx;
    }
    const double q_unit = unit_q * inv_dx;  // charge units to density in one cell
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int it = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); it < S.n_items; it += warps) {
        const WorkItem I = S.items[it];
        const double q_sheet = (double)(S.seg_q ? I.qh : 2 * I.qh) * q_unit;
        const int l0 = lane * R;
        unsigned u[R + 1];
        float v[R + 1];
        int q[R + 1];
        const int mine = max(0, min(R, I.count - l0));  // tracers of this lane
#pragma unroll
        for (int r = 0; r < R; ++r) {
            u[r] = 0u;
            v[r] = 0.f;
            q[r] = I.qh;
        }
        if (mine == R) {
            static_assert(R % 4 == 0, "a lane's tracers load as 16-byte vectors");
#pragma unroll
            for (int k = 0; k < R / 4; ++k) {
                const uint4 a = reinterpret_cast<const uint4 *>(U + I.t0 + l0)[k];
                const float4 b = reinterpret_cast<const float4 *>(V + I.t0 + l0)[k];
                u[4 * k] = a.x, u[4 * k + 1] = a.y, u[4 * k + 2] = a.z, u[4 * k + 3] = a.w;
                v[4 * k] = b.x, v[4 * k + 1] = b.y, v[4 * k + 2] = b.z, v[4 * k + 3] = b.w;
                if (Qh) {
                    const int4 c = reinterpret_cast<const int4 *>(Qh + I.t0 + l0)[k];
                    q[4 * k] = c.x, q[4 * k + 1] = c.y, q[4 * k + 2] = c.z, q[4 * k + 3] = c.w;
                }
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (r < mine) {
                    u[r] = U[I.t0 + l0 + r];
                    v[r] = V[I.t0 + l0 + r];
                    if (Qh)
                        q[r] = Qh[I.t0 + l0 + r];
                }
        }
        // the tracer after the lane's last one: the next lane's first, or
        // (the item's last lane) the halo
        unsigned ue = __shfl_down_sync(0xffffffffu, u[0], 1);
        float ve = __shfl_down_sync(0xffffffffu, v[0], 1);
        int qe = __shfl_down_sync(0xffffffffu, q[0], 1);
        int segs = mine;
        if (mine > 0 && l0 + mine == I.count) {
            if (I.halo >= 0) {
                ue = U[I.halo] + I.halo_shift;
                ve = V[I.halo];
                qe = Qh ? Qh[I.halo] : I.qh;
            } else {
                --segs;
            }
        }
#pragma unroll
        for (int r = 1; r <= R; ++r)
            if (r == mine) {
                u[r] = ue;
                v[r] = ve;
                q[r] = qe;
            }
        MomentRun<W> run(n, j, nx);
        auto wrap = [&](int c) {
            while (c >= nx)
                c -= nx;
            return c;
        };
#pragma unroll 1
        for (int r = 0; r < R; ++r) {
            unsigned ua = u[0], ub = u[1];
            float fa = v[0], fb = v[1];
            int qa = q[0], qb = q[1];
#pragma unroll
            for (int k = 1; k < R; ++k)
                if (k == r) {
                    ua = u[k], ub = u[k + 1];
                    fa = v[k], fb = v[k + 1];
                    qa = q[k], qb = q[k + 1];
                }
            // the cells (first order: nodes) between the ends: `between` of
            // them from `next` on get dens each, and d0, d0 + d1, ... of j
            int between = 0, next = 0;
            double dens = 0.0, d0 = 0.0, d1 = 0.0;
            if (r < segs) {
                const long long span = seg_span(ua, ub, nx4);
                const bool back = span < 0;
                const unsigned long long len = (unsigned long long)(back ? -span : span);
                const unsigned long long a = (unsigned long long)cell_coord(back ? ub : ua, nx);
                const unsigned long long b = a + len;
                const int jl = (int)(a >> 32), cuts = (int)(b >> 32) - jl;
                // fractions of their cells at the lower and upper end
                const double f0 = W || cuts ? cells_double((unsigned)a) : 0.0;
                const double f1 = W || cuts ? cells_double((unsigned)b) : 0.0;
                double va = widen(fa), vb = widen(fb);
                double qs = q_sheet, vbar = 0.0;
                if (Qh)
                    qs = cells_double((unsigned long long)(unsigned)(S.seg_q ? qa : qa + qb)) * (q_unit * 0x1p32);
                if (W == 0 || len == 0) {
                    if (Qh && qa + qb > 0) {
                        const double x = cells_double((unsigned)(qa + qb));
                        vbar = (cells_double((unsigned)qa) * va + cells_double((unsigned)qb) * vb) *
                               cells_recip((unsigned)(qa + qb), x) * unit_v;
                    } else {
                        vbar = (va + vb) * (0.5 * unit_v);
                    }
                }
                double inv = 0.0;
                if (cuts > 0) {
                    inv = cells_recip(len, cells_double(len));
                    dens = qs * inv;  // charge per cell
                }
                double ln[W + 1], lj[W + 1];  // the lower end's cell gets (first order: its two nodes)
                double hn[W + 1], hj[W + 1];  // the upper end's, if it is another
                if (W == 0) {
                    ln[0] = qs;
                    if (cuts > 0) {
                        ln[0] = dens * (1.0 - f0);
                        hn[0] = dens * f1;
                        hj[0] = hn[0] * vbar;
                        d0 = dens * vbar;
                        between = cuts - 1;
                        next = jl + 1;
                    }
                    lj[0] = ln[0] * vbar;
                } else {
                    // a piece of charge p between the fractions s0 and s1 of a
                    // cell, its velocity from u0 to u1: the upper node weighs
                    // s, the lower one 1 - s.  (A point is such a piece too.)
                    double vl = (back ? vb : va) * unit_v, vr = (back ? va : vb) * unit_v;
                    if (len == 0)
                        vl = vr = vbar;
                    double s1 = f1, u1 = vr, p = qs, dv = 0.0;
                    if (cuts > 0) {
                        dv = (vr - vl) * inv;  // velocity gained per cell
                        s1 = 1.0;
                        u1 = fma(1.0 - f0, dv, vl);
                        p = dens * (1.0 - f0);
                    }
                    const double h = 0.5 * p, t = vl + u1;
                    ln[W] = h * (f0 + s1);
                    ln[0] = p - ln[W];
                    lj[W] = h * (1.0 / 3.0) * fma(f0, t + vl, s1 * (t + u1));
                    lj[0] = fma(h, t, -lj[W]);
                    if (cuts > 0) {
                        const double u0 = fma(-f1, dv, vr);  // at the upper end's cell's edge
                        const double g = dens * f1, hh = 0.5 * g, tt = u0 + vr;
                        hn[W] = hh * f1;
                        hn[0] = g - hn[W];
                        hj[W] = hh * (1.0 / 3.0) * f1 * (tt + vr);
                        hj[0] = fma(hh, tt, -hj[W]);
                        if (cuts > 1) {
                            // the outer halves of the whole cells between
                            const double hd = 0.5 * dens, sixth = dv * (1.0 / 3.0);
                            ln[W] += hd;
                            lj[W] = fma(hd, u1 + sixth, lj[W]);
                            hn[0] += hd;
                            hj[0] = fma(hd, u0 - sixth, hj[0]);
                            between = cuts - 2;
                            next = jl + 2;
                            d1 = dens * dv;
                            d0 = fma(dens, u1, d1);
                        }
                    }
                }
                // the end that the sheet reaches last goes last: the next
                // particle starts in its cell
                const int jr = wrap(jl + cuts);
                if (cuts == 0) {
                    run.add(jl, ln, lj);
                } else if (back) {
                    run.add(jr, hn, hj);
                    run.add(jl, ln, lj);
                } else {
                    run.add(jl, ln, lj);
                    run.add(jr, hn, hj);
                }
                next = wrap(next);
                if (between < kMomentCells) {
                    for (int k = 0; k < between; ++k) {
                        atomicAdd(n + next, dens);
                        atomicAdd(j + next, d0);
                        if (W == 1)
                            d0 += d1;
                        next = next + 1 == nx ? 0 : next + 1;
                    }
                    between = 0;
                }
            }
            // many cells between: one particle after another, over the lanes
            unsigned who = __ballot_sync(0xffffffffu, between > 0);
            while (who) {
                const int from = __ffs(who) - 1;
                who &= who - 1u;
                const int cells = __shfl_sync(0xffffffffu, between, from), at = __shfl_sync(0xffffffffu, next, from);
                const double dn = __shfl_sync(0xffffffffu, dens, from), dj = __shfl_sync(0xffffffffu, d0, from);
                const double dd = W == 1 ? __shfl_sync(0xffffffffu, d1, from) : 0.0;
                for (int k = lane; k < cells; k += 32) {
                    const int c = wrap(at + k);
                    atomicAdd(n + c, dn);
                    atomicAdd(j + c, W == 1 ? fma(cells_double((unsigned long long)(unsigned)k << 32), dd, dj) : dj);
                }
            }
        }
        run.flush();
    }
}

// The sums of the copies of n and j, in order
__global__ void __launch_bounds__(256) k_moments_sum(int nx, const double *scratch, double *n, double *j, int copies)
{
    const int c = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (c >= nx)
        return;
    const double *cn = scratch + c, *cj = cn + nx;
    double sn = 0.0, sj = 0.0;
#pragma unroll 8
    for (int k = 0; k < copies; ++k) {
        sn += cn[(size_t)k * 2 * nx];
        sj += cj[(size_t)k * 2 * nx];
    }
    n[c] = sn;
    j[c] = sj;
}

}  // namespace

// On a small mesh all atomics meet in a few slices of the L2 (one 80 % busy,
// the average 7 %: 229 and 298 us for the two orders on 512 cells), so blocks take turns with copies of n and j, kMomentWords
// cells altogether, in the caller's scratch: no block shares a copy with all
// others.  Not for few items (a block for every copy) and without scratch.
constexpr int kMomentWords = 16384;

int moment_copies(int nx, long long n_items)
{
    return (int)std::max(1ll, std::min<long long>(kMomentWords / nx, (n_items + 7) / 8));
}

cudaError_t launch_moments(const SimDev &sim, double *scratch, int copies, int weighting, double box_length,
                           double unit_q, double unit_v, double *n, double *j, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    if (copies > 1) {
        e = cudaMemsetAsync(scratch, 0, 2 * sizeof(double) * (size_t)copies * (size_t)sim.nx, s);
    } else {
        e = cudaMemsetAsync(n, 0, sizeof(double) * (size_t)sim.nx, s);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(j, 0, sizeof(double) * (size_t)sim.nx, s);
    }
    if (e != cudaSuccess)
        return e;
    // one warp per work item
    constexpr int warps = kMomentThreads / 32;
    const int grid =
        (int)std::max<long long>(1, std::min<long long>(131072 / warps, ((long long)sim.n_items + warps - 1) / warps));
    const double inv_dx = (double)sim.nx / box_length;
    if (weighting == 0)
        k_moments<0><<<grid, kMomentThreads, 0, s>>>(sim, inv_dx, unit_q, unit_v, n, j, scratch, copies);
    else
        k_moments<1><<<grid, kMomentThreads, 0, s>>>(sim, inv_dx, unit_q, unit_v, n, j, scratch, copies);
    count_launches(1);
    if (copies > 1) {
        k_moments_sum<<<(sim.nx + 255) / 256, 256, 0, s>>>(sim.nx, scratch, n, j, copies);
        count_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace sic

namespace sic {
namespace {

// ---------------------------------------------------------- refinement ----
// Sec. 2.6: a particle longer than the refinement length (lfix, position
// units) gets a new tracer at its centre.  k_refine_count counts those
// particles per work item; k_refine_scatter writes every tracer, and after
// each split particle's first tracer the new one, into the new layout, with
// per-particle charges: each half of a split particle gets half its charge
// (the first floor(Q / 2), the second the rest).  One thread per work item.
__device__ __forceinline__ bool refine_seg(const WorkItem &W, long long t, const unsigned *U, long long &d,
                                           long long &t1)
{
    const long long last = W.t0 + W.count - 1;
    unsigned shift = 0u;
    t1 = t + 1;
    if (t == last) {
        if (W.halo < 0)
            return false;
        t1 = W.halo;
        shift = W.halo_shift;
    }
    d = (long long)(int)(U[t1] + shift - U[t]);
    return true;
}

__global__ void k_refine_count(const SimDev S, long long lfix, int32_t *splits)
{
    const unsigned *U = S.U[S.sc->buf & 1];
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < S.n_items; it += gridDim.x * blockDim.x) {
        const WorkItem W = S.items[it];
        int c = 0;
        for (long long t = W.t0; t < W.t0 + W.count; ++t) {
            long long d, t1;
            if (refine_seg(W, t, U, d, t1) && (d > lfix || -d > lfix))
                ++c;
        }
        splits[it] = c;
    }
}

__global__ void k_refine_scatter(const SimDev S, long long lfix, const int64_t *out_base, uint32_t *U2, float *V2,
                                 int32_t *Q2)
{
    const int b = (int)(S.sc->buf & 1);
    const unsigned *U = S.U[b];
    const float *V = S.V[b];
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < S.n_items; it += gridDim.x * blockDim.x) {
        const WorkItem W = S.items[it];
        long long out = out_base[it];
        for (long long t = W.t0; t < W.t0 + W.count; ++t) {
            long long d = 0, t1 = t;
            const bool seg = refine_seg(W, t, U, d, t1);
            // the particle's charge: its own (refined sheets), else the
            // mean of its tracers' weights (the sheet's, or per tracer)
            const int Q = !seg ? 0 : S.seg_q ? S.Qh[t] : S.Qh ? S.Qh[t] + S.Qh[t1] : 2 * W.qh;
            U2[out] = U[t];
            V2[out] = V[t];
            if (seg && (d > lfix || -d > lfix)) {
                Q2[out] = Q >> 1;
                ++out;
                U2[out] = U[t] + (unsigned)(int)(d >> 1);  // floor of half the segment
                V2[out] = 0.5f * (V[t] + V[t1]);
                Q2[out] = Q - (Q >> 1);
            } else {
                Q2[out] = Q;
            }
            ++out;
        }
    }
}

}  // namespace

cudaError_t launch_refine_count(const SimDev &sim, long long lfix, int32_t *splits, cudaStream_t s)
{
    const int grid = (int)std::max<long long>(1, std::min<long long>(4096, ((long long)sim.n_items + 255) / 256));
    k_refine_count<<<grid, 256, 0, s>>>(sim, lfix, splits);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_refine_scatter(const SimDev &sim, long long lfix, const int64_t *out_base, uint32_t *U2, float *V2,
                                  int32_t *Q2, cudaStream_t s)
{
    const int grid = (int)std::max<long long>(1, std::min<long long>(4096, ((long long)sim.n_items + 255) / 256));
    k_refine_scatter<<<grid, 256, 0, s>>>(sim, lfix, out_base, U2, V2, Q2);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace sic
