// sic_run.cu -- k_run: many steps of one or many simulations in one
// cooperative launch (sic_step, sic_run, batches and the server take it where
// a step is short; k_step of sic_kernels.cu has one launch a step).
#include <mutex>

#include "sic_item.cuh"

namespace sic {

namespace {

// ------------------------------------------------- many steps a launch ----

// A bounded wait until *bar reaches target (modulo 2^32): false after this many
// polls (a poll is a trip to L2, about 0.7 us).
__device__ __forceinline__ bool group_wait(const unsigned *bar, unsigned target, int polls)
{
    for (int i = 0; i < polls; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if ((int)(v - target) >= 0)
            return true;
    }
    return false;
}

// n_steps steps of every simulation of the launch, without going back to the
// host or starting a new grid in between: a step of a small simulation is a
// chain of latencies, and launching it (claims, descriptors, the last block's
// field solve while the others are gone, the next grid's start) was most of
// it.  The blocks of the grid are split into one group per simulation
// (A.block_begin), all resident at once (a cooperative launch), and the groups
// do not wait for one another.  The warps of a group take the simulation's
// items in turn, always the same ones, so nothing is claimed.  A step:
//   1. push and deposit the warp's items (do_item, as in k_step);
//   2. add the block's mesh and sums into the step's buffers with atomics and
//      wait until all blocks of the group have;
//   3. every block solves the field from the whole mesh for itself (the same
//      integers, so the same bits), the first item of the next step already on
//      its way; the group's last block also records the step.
// A group of one block keeps the mesh in shared memory.  The mesh and the
// sums have three buffers: the one of step i is cleared during step i + 2,
// when every block has read it.  The second and third mesh are the plan's own:
// nothing that a call reading the simulation on another stream writes is theirs.
//
// us per step in runs of 160 steps, graphs of single steps and this: 4 K
// tracers 9.8 and 6.3, 262 K 10.8 and 5.7, 430 K irregular 28 and 16, 8.4 M 41
// and 36; piecewise linear 0.5 M 72 and 42, first order 0.5 M 20.7 and 10.3.
// Folded 2.3 M and 4.2 M go from 33.8 to 32.1 and from 50.6 to 46.1 (bound by
// the deposit).  Up to one item a warp (622 K tracers) the tracers never leave
// shared memory between the first step and the last: with their copies 262 K
// took 7.1, first order 12.6.  What is left of a small step (262 K: about 2 us
// the items, 3 the adds into L2 and the wait, 1.5 the field) are latencies.
template <bool PER_Q, bool GEN>
__device__ __forceinline__ void run_steps(const RunArgs &A, int slot)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Shared &sh = *reinterpret_cast<Shared *>(smem);
    const int nx_max = A.nx_max;
    unsigned long long *mesh_region = reinterpret_cast<unsigned long long *>(smem + kSharedHead);
    Hist hist;
    hist.lo = reinterpret_cast<unsigned *>(mesh_region);
    hist.hi = hist.lo + nx_max;
    Hist diff;
    diff.lo = reinterpret_cast<unsigned *>(mesh_region + nx_max);
    diff.hi = diff.lo + nx_max + 2;
    float2 *ek = reinterpret_cast<float2 *>(mesh_region + nx_max + nx_max + 2);
    char *stage_base = reinterpret_cast<char *>(smem) + stage_offset(nx_max);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    char *my_stage = stage_base + (size_t)warp * WarpBuf<PER_Q, true>::bytes;
    unsigned short *tasks =
        reinterpret_cast<unsigned short *>(stage_base + (size_t)NW * WarpBuf<PER_Q, true>::bytes) + warp * WT;

    const int rank = (int)blockIdx.x - A.block_begin[slot];
    const int G = A.block_begin[slot + 1] - A.block_begin[slot];
    const bool recorder = rank == G - 1;
    RunCtl *ctl = A.ctl + slot;

    for (int i = tid; i < (int)(sizeof(SimDev) / 4); i += B)
        reinterpret_cast<unsigned *>(&sh.sim)[i] = reinterpret_cast<const unsigned *>(A.sims + slot)[i];
    if (tid < 2 * NW)
        mbar_init(&sh.mbar[tid >> 1][tid & 1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    const SimDev &S = sh.sim;
    const int nx = S.nx, n_items = S.n_items;
    const WorkItem *items = S.items;
    for (int j = tid; j < nx; j += B) {
        hist.lo[j] = 0u;
        hist.hi[j] = 0u;
        ek[j] = __ldcg(S.Ek + j);
    }
    for (int j = tid; j < nx + 2; j += B) {
        diff.lo[j] = 0u;
        diff.hi[j] = 0u;
    }
    if (tid == 0) {
        sh.diff_used = 0;
        sh.ke[0] = sh.ke[1] = sh.p[0] = sh.p[1] = 0ull;
        sh.step_err = 0u;
        sh.gave_up = 0u;
        sh.hold = __ldcg(&S.sc->hold);
        sh.buf = __ldcg(&S.sc->buf);
        sh.pre_err = __ldcg(&S.sc->err);
        sh.pre_step = __ldcg(&S.sc->step);
        sh.pre_we = __ldcg(&S.sc->we);
        sh.pre_wk = __ldcg(&S.sc->wk);
    }
    __syncthreads();
    // a held simulation stays as it is; every block of the group sees the same
    // word (the recorder writes it after all of them have been counted)
    const unsigned hold0 = sh.hold;
    if (hold0)
        return;
    unsigned err = sh.pre_err;
    int src = (int)(sh.buf & 1u);
    const long long step0 = sh.pre_step;
    int row_slot = (int)(step0 % S.hist_len);  // the recorder's next row
    const bool track_all = S.refine_seg > 0 && S.refine_seg < (1ll << 16);  // refinement below a cell
    const int32_t *Qh = S.Qh;
    const int stride = G * NW, first = warp * G + rank;
    // The first three quarters of the rounds are the warp's own items (first,
    // first + stride, ...); the rest are claimed one at a time, an item ahead,
    // since folded and quiet sheets differ by a factor of three.
    const int rounds = (n_items + stride - 1) / stride;
    const bool claims = G > 1 && rounds > 1;
    const int own = claims ? max(1, rounds * 3 / 4) : rounds;
    unsigned claimed = 0;  // lane 0: the claim in flight

    unsigned phase = 0;
    int s = 0;
    bool timed_out = false;
    // A simulation of at most one item a warp is kept: the items stay in their
    // stages from the first step to the last, which writes them back in place.
    const bool kept = rounds == 1;
    const bool busy = first < n_items;
    if (busy && lane == 0) {
        desc_fetch(&sh.own[warp], items + first);
        desc_wait();
        stage_issue<PER_Q>(sh.own[warp], S.U[src], S.V[src], Qh, my_stage, &sh.mbar[warp][0]);
        if (claims && own == 1)
            claimed = atomicAdd(&ctl->cursor[0], 1u);
    }
    __syncwarp();
    if (kept && busy) {
        const WorkItem W = sh.own[warp];
        Beside &b = sh.beside[warp];
        if (lane == 0 && W.halo >= 0) {
            b.hu = __ldcg(S.U[src] + W.halo);
            b.hv = __ldcg(S.V[src] + W.halo);
            if (PER_Q)
                b.hq = Qh[W.halo];
        }
        if (GEN && S.pl != nullptr && lane == 1) {
            const WorkItemPL P = S.pl[first];
            if (P.prev >= 0) {
                b.pu = __ldcg(S.U[src] + P.prev);
                b.pv = __ldcg(S.V[src] + P.prev);
                if (PER_Q)
                    b.pq = Qh[P.prev];
            }
            if (P.next2 >= 0) {
                b.nu = __ldcg(S.U[src] + P.next2);
                b.nv = __ldcg(S.V[src] + P.next2);
                if (PER_Q)
                    b.nq = Qh[P.next2];
            }
        }
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&sh.mbar[warp][0], 0u))) {
            timed_out = true;
            mbar_drain(&sh.mbar[warp][0], 0u);
        }
        __syncwarp();
    }

    // The recorder's last warp: the row of the step whose sums (the words of
    // several blocks, in sh.pre) and field sums it has put aside.  Lane 0 the
    // kinetic energy, lane 1 the momentum (the same arithmetic side by side),
    // lane 2 the rest.
    auto record = [&]() {
        double *row = S.hist + 4 * (size_t)row_slot;
        if (lane < 2) {
            unsigned long long lo, hi;
            if (G > 1) {
                const unsigned long long *l = sh.pre + 4 * lane;
                const unsigned __int128 u = (unsigned __int128)l[0] + ((unsigned __int128)l[1] << 32) +
                                            ((unsigned __int128)l[2] << 64) + ((unsigned __int128)l[3] << 96);
                lo = (unsigned long long)u;
                hi = (unsigned long long)(u >> 64);
            } else {
                lo = sh.tot[lane][0];
                hi = sh.tot[lane][1];
            }
            row[1 + lane] = (lane ? S.p_scale : S.ke_scale) *
                            times_pow2(i128_words_to_double(lo, hi), -(lane ? S.p_u : S.ke_u));
        } else if (lane == 2) {
            row[0] = sh.pre_we;
            row[3] = (double)(long long)sh.pre[8];
            double w = 0.0;
#pragma unroll
            for (int i = 0; i < NW; ++i)
                w += sh.da[i];
            w *= S.we_scale;
            double wk = sh.pre_wk;
            const int mode_k = S.mode_k;
            if (mode_k) {
                // W_k = dx / nx |E^_k|^2 (half at k = nx/2) = (2 or 1) / nx we_scale |Z|^2
                double re = 0.0, im = 0.0;
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    re += (double)sh.mre[i];
                    im += (double)sh.mim[i];
                }
                S.mhist[row_slot] = wk;
                wk = (2 * mode_k == nx ? 1.0 : 2.0) / nx * S.we_scale * (re * re + im * im);
            }
            sh.pre_we = w;
            sh.pre_wk = wk;
        }
        row_slot = row_slot + 1 == S.hist_len ? 0 : row_slot + 1;
    };

    for (int st = 0;; ++st) {
        const int now = st % 3, nxt_buf = (st + 1) % 3;
        auto mesh_of = [&](int k) {
            return k == 0 ? S.mesh : S.run_mesh[k - 1];
        };
        if (G > 1 && recorder) {
            unsigned long long *m = mesh_of(nxt_buf);
            for (int j = tid; j < nx; j += B)
                m[j] = 0ull;
            if (tid < (int)(sizeof(SimAccum) / 8))
                reinterpret_cast<unsigned long long *>(&ctl->acc[nxt_buf])[tid] = 0ull;
            if (tid == 32)
                ctl->cursor[nxt_buf] = 0u;
        }
        // ---- 1. items
        const unsigned *Uin = S.U[src];
        const float *Vin = S.V[src];
        unsigned *Uout = S.U[src ^ 1];
        float *Vout = S.V[src ^ 1];
        unsigned rerr = 0, mseg = 0, mlen = 0;
        long long ake = 0, ap = 0;
        if (kept && busy && !timed_out) {
            const WorkItem W = sh.own[warp];
            const WorkItemPL *plw = (GEN && S.pl != nullptr) ? S.pl + first : nullptr;
            char *tab = my_stage + WarpBuf<PER_Q, true>::stage;
            auto mid = []() {};
            if (W.count == WT)
                do_item<true, true, PER_Q, true, true, GEN, true>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh, nx, 1.0f, 1,
                                                                 rerr, my_stage, tab, tasks, ake, ap, mseg, mlen, plw,
                                                                 S.deposit, S.seg_q, track_all, mid);
            else
                do_item<true, true, PER_Q, false, true, GEN, true>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh, nx, 1.0f,
                                                                  1, rerr, my_stage, tab, tasks, ake, ap, mseg, mlen, plw,
                                                                  S.deposit, S.seg_q, track_all, mid);
        }
        for (int i = kept ? -1 : first, r = 0; i >= 0 && i < n_items; ++r) {
            int nxt;
            if (r + 1 < own)
                nxt = i + stride;
            else if (claims)
                nxt = own * stride + (int)__shfl_sync(0xffffffffu, claimed, 0);
            else
                nxt = n_items;
            nxt = nxt < n_items ? nxt : -1;
            if (claims && r + 2 >= own && nxt >= 0 && lane == 0)
                claimed = atomicAdd(&ctl->cursor[now], 1u);
            const WorkItem W = r == 0 ? sh.own[warp] : sh.desc[warp][s].w;
            const WorkItemPL *plw = (GEN && S.pl != nullptr) ? S.pl + i : nullptr;
            if (nxt >= 0 && lane == 0)
                desc_fetch(&sh.desc[warp][s ^ 1].w, items + nxt);
            const bool ok = mbar_wait_bounded(&sh.mbar[warp][s], (phase >> s) & 1u);
            phase ^= 1u << s;
            if (!__all_sync(0xffffffffu, ok)) {  // give up (the next item's copies have not started)
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
            char *stg = my_stage + s * WarpBuf<PER_Q, true>::stage;
            if (W.count == WT)
                do_item<true, true, PER_Q, true, true, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh, nx, 1.0f, 1,
                                                           rerr, stg, stg, tasks, ake, ap, mseg, mlen, plw, S.deposit, S.seg_q,
                                                           track_all, mid);
            else
                do_item<true, true, PER_Q, false, true, GEN, false>(W, Uin, Vin, Uout, Vout, Qh, ek, hist, diff, sh, nx, 1.0f, 1,
                                                            rerr, stg, stg, tasks, ake, ap, mseg, mlen, plw, S.deposit,
                                                            S.seg_q, track_all, mid);
            __syncwarp();
            s ^= 1;
            i = nxt;
        }

        // ---- 2. the block's mesh and sums
        const Acc128 k2 = i64_warp_sum(ake);
        const Acc128 p2 = i64_warp_sum(ap);
        mseg = max(mseg, (unsigned)(((unsigned long long)mlen * (unsigned)(nx << SIC_POS_WIND_BITS)) >> 16));
        mseg = __reduce_max_sync(0xffffffffu, mseg);
        if (lane == 0) {
            sh.wke[warp][0] = (long long)k2.lo;
            sh.wke[warp][1] = k2.hi;
            sh.wp[warp][0] = (long long)p2.lo;
            sh.wp[warp][1] = p2.hi;
            sh.wmseg[warp] = mseg;
        }
        {
            const unsigned bad = (rerr >> 30 ? SIC_ERR_RANGE : 0u) | (timed_out ? SIC_ERR_TIMEOUT : 0u);
            if (bad)
                atomicOr(&sh.step_err, bad);
        }
        if (!kept)  // the new positions and velocities are read by the next step's bulk copies
            asm volatile("fence.proxy.async;" ::: "memory");
        __syncthreads();
        const bool diffs = sh.diff_used != 0;
        if (diffs)
            add_diff_prefix(hist, diff, nx, sh);
        if (warp == 1 || warp == 2) {
            // the block's sums: lanes 0..7 hold the warps'
            const long long (*w)[2] = warp == 1 ? sh.wke : sh.wp;
            Acc128 t{0ull, 0ll};
            if (lane < NW)
                t = Acc128{(unsigned long long)w[lane][0], w[lane][1]};
#pragma unroll
            for (int o = NW / 2; o > 0; o >>= 1) {
                Acc128 b;
                b.lo = __shfl_down_sync(0xffffffffu, t.lo, o);
                b.hi = __shfl_down_sync(0xffffffffu, t.hi, o);
                acc_add(t, b);
            }
            if (lane == 0) {
                unsigned long long *spill = warp == 1 ? sh.ke : sh.p;
                acc_add(t, Acc128{spill[0], (long long)spill[1]});
                spill[0] = spill[1] = 0ull;
                if (G > 1) {
                    unsigned long long *to = warp == 1 ? ctl->acc[now].ke : ctl->acc[now].p;
                    const unsigned l[4] = {(unsigned)t.lo, (unsigned)(t.lo >> 32), (unsigned)t.hi,
                                           (unsigned)((unsigned long long)t.hi >> 32)};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (l[i])
                            atomicAdd(to + i, (unsigned long long)l[i]);
                } else {
                    sh.tot[warp - 1][0] = t.lo;
                    sh.tot[warp - 1][1] = (unsigned long long)t.hi;
                }
            }
        } else if (warp == 3) {
            const unsigned m = __reduce_max_sync(0xffffffffu, lane < NW ? sh.wmseg[lane] : 0u);
            if (lane == 0) {
                if (G > 1) {
                    if (m)
                        atomicMax(&ctl->acc[now].maxseg, (unsigned long long)m);
                    if (sh.step_err)
                        atomicOr(&ctl->acc[now].pad[0], (unsigned long long)sh.step_err);
                } else {
                    sh.step_mseg = m;
                }
            }
        }
        unsigned long long *mesh = mesh_of(now);
        if (G > 1) {
            for (int j = tid; j < nx; j += B) {
                const unsigned long long h = hist.get(j);
                if (h)
                    atomicAdd(mesh + j, h);
            }
            __threadfence();
            __syncthreads();
            if (recorder && warp == NW - 1 && st > 0)
                record();  // the step before's
            if (tid == 0) {
                atomicAdd(&ctl->bar, 1u);
                if (group_wait(&ctl->bar, (unsigned)(st + 1) * (unsigned)G, A.wait_polls)) {
                    sh.step_mseg = __ldcg(&ctl->acc[now].maxseg);
                    sh.step_err = (unsigned)__ldcg(&ctl->acc[now].pad[0]);
                } else {
                    sh.gave_up = 1u;
                }
            }
        }
        __syncthreads();
        if (sh.gave_up) {
            // (No copies are in flight: the next step's have not started.)  The
            // bits stay whatever the recorder does, which may still see the
            // count complete and record this step: this block's part of the
            // state is missing, so the simulation is not stepped again, and
            // the group's buffers, which nobody clears now, are not used again.
            if (tid == 0) {
                atomicOr(&S.sc->err, SIC_ERR_TIMEOUT);
                atomicOr(&S.sc->hold, SIC_HOLD_ERROR);
            }
            return;
        }
        // hold the simulation when it needs the host (the rules of
        // field_epilogue): every block decides the same
        const long long mm = (long long)sh.step_mseg;
        err |= sh.step_err;
        if (S.strict && mm > ((long long)nx << 16))
            err |= SIC_ERR_SEGLONG;
        if (mm >= ((long long)(3 * nx) << 15))
            err |= SIC_ERR_RANGE;
        unsigned hold = err ? SIC_HOLD_ERROR : 0u;
        if (S.refine_seg > 0 && mm > S.refine_seg)
            hold |= SIC_HOLD_REFINE;
        const bool last = hold || st + 1 == A.n_steps;
        if (!kept)
            src ^= 1;
        // the next step's first item comes in during the field solve
        auto next_item = [&]() {
            if (!kept && !last && busy && lane == 0) {
                asm volatile("fence.proxy.async;" ::: "memory");
                stage_issue<PER_Q>(sh.own[warp], S.U[src], S.V[src], Qh, my_stage + s * WarpBuf<PER_Q, true>::stage,
                                   &sh.mbar[warp][s]);
                if (claims && own == 1)
                    claimed = atomicAdd(&ctl->cursor[nxt_buf], 1u);
            }
        };
        if (last && !recorder)
            break;

        // ---- 3. the field (field_epilogue's integers and its order of FP32 sums)
        unsigned long long limb = 0ull;  // the recorder's last warp: the step's sums
        if (recorder && warp == NW - 1 && lane < 8)
            limb = G > 1 ? __ldcg(lane < 4 ? &ctl->acc[now].ke[lane] : &ctl->acc[now].p[lane - 4]) : 0ull;
        const int per = (nx + B - 1) / B;
        const int j0 = min(tid * per, nx), j1 = min(j0 + per, nx);
        long long lsum = 0;
        __int128 m1 = 0;  // sum_j j mesh_j over this thread's cells
        for (int j = j0; j < j1; j += 4) {
            unsigned long long mv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                mv[k] = j + k < j1 ? (G > 1 ? __ldcg(mesh + j + k) : hist.get(j + k)) : 0ull;
            if (j == j0)
                next_item();
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (j + k < j1) {
                    if (G > 1)
                        hist.set(j + k, mv[k]);
                    lsum += (long long)mv[k];
                    m1 += (__int128)(j + k) * (long long)mv[k];
                }
        }
        if (j0 == j1)  // (a thread without a cell)
            next_item();
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
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w < warp)
                before += sh.w64[w];
            qtot += sh.w64[w];
            M1 += make_i128(sh.hi[w], sh.lo[w]);
        }
        const __int128 sumD = (__int128)((long long)nx * (nx - 1) / 2) * qtot - (__int128)nx * M1;
        // K_j = nx D_j - sumD, from cell to cell K_{j+1} = K_j + nx^2 mesh_j - nx Q
        __int128 K = (__int128)nx * ((__int128)nx * (incl - lsum + before) - (__int128)j0 * qtot) - sumD;
        const long long nx2 = (long long)nx * nx;
        const __int128 nxq = (__int128)nx * qtot;
        const bool nodes = GEN && S.deposit == SIC_DEPOSIT_FIRST;
        const int mode_k = recorder ? S.mode_k : 0;
        float wloc = 0.f, mre = 0.f, mim = 0.f;
#pragma unroll 1
        for (int j = j0; j < j1; ++j) {
            const long long m = (long long)hist.get(j);
            const __int128 Kn = K + (__int128)nx2 * m - nxq;
            const Norm128 nk = norm128(nodes ? K + Kn : K);
            ek[j].x = __fmul_rn(norm_to_float(nk, S.ek_exp - (nodes ? 1 : 0)), S.ek_mant);
            if (recorder) {
                const float kn = norm_to_float(nk, nodes ? -61 : -60);
                wloc = __fmaf_rn(kn, kn, wloc);
                if (mode_k)
                    mode_add(kn, j, mode_k, nx, mre, mim);
                if (last)
                    S.mesh_last[j] = m;
            }
            hist.lo[j] = 0u;
            hist.hi[j] = 0u;
            K = Kn;
        }
        if (diffs)
            for (int j = tid; j < nx + 2; j += B) {
                diff.lo[j] = 0u;
                diff.hi[j] = 0u;
            }
        if (recorder) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                wloc = __fadd_rn(wloc, __shfl_down_sync(0xffffffffu, wloc, o));
            if (lane == 0)
                sh.da[warp] = (double)wloc;
            if (warp == NW - 1 && lane < 9)
                sh.pre[lane] = lane < 8 ? limb : (unsigned long long)qtot;
            __syncwarp();
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
        }
        if (tid == 0) {
            sh.diff_used = 0;
            sh.step_err = 0u;
        }
        __syncthreads();
        for (int j = tid; j < nx; j += B) {
            const int jn = (j + 1 == nx) ? 0 : j + 1;
            const float e0 = ek[j].x, de = ek[jn].x - e0;
            ek[j].y = de;
            if (last)
                S.Ek[j] = make_float2(e0, de);
        }
        __syncthreads();
        // The row: 900 cycles of FP64 that the next step's items would start
        // late by, so of several blocks the recorder writes it while it waits
        // for the others (4096 tracers on 64 cells, 500 steps: 3.17 to 2.97 ms)
        if (recorder && warp == NW - 1 && (G == 1 || last)) {
            record();
            if (lane == 2 && last) {
                SimScalars *sc = S.sc;
                sc->we = sh.pre_we;
                sc->wk = sh.pre_wk;
                sc->step = step0 + st + 1;
                sc->q_total = qtot;
                sc->maxseg = mm;
                if (err)  // (added: a block that gave up has put its own there)
                    atomicOr(&sc->err, err);
                if (hold)
                    atomicOr(&sc->hold, hold);
                sc->buf = (unsigned)src;
            }
        }
        if (last)
            break;
    }
    if (kept && busy && !timed_out) {
        // the item back where it came from
        const WorkItem W = sh.own[warp];
        const int l0 = lane * R, mine = min(R, W.count - l0);
        const unsigned *bu = reinterpret_cast<const unsigned *>(my_stage) + l0;
        const float *bv = reinterpret_cast<const float *>(my_stage + kStageBytesU) + l0;
        unsigned *U = S.U[src] + W.t0 + l0;
        float *V = S.V[src] + W.t0 + l0;
        if (mine == R) {
#pragma unroll
            for (int k = 0; k < R / 4; ++k) {
                reinterpret_cast<uint4 *>(U)[k] = reinterpret_cast<const uint4 *>(bu)[k];
                reinterpret_cast<float4 *>(V)[k] = reinterpret_cast<const float4 *>(bv)[k];
            }
        } else {
            for (int r = 0; r < mine; ++r) {
                U[r] = bu[r];
                V[r] = bv[r];
            }
        }
    }
    if (G == 1)
        return;
    // Leave the mesh, the sums and the block count clear for the next launch.
    // The last block out does it: until a block is counted here it may still
    // be reading the last step's sums, and the recorder its mesh.
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        sh.last_out = atomicAdd(&ctl->out, 1u) + 1 == (unsigned)G;
    }
    __syncthreads();
    if (!sh.last_out)
        return;
    for (int j = tid; j < nx; j += B)
        S.mesh[j] = 0ull;
    for (int i = tid; i < (int)(sizeof(ctl->acc) / 8); i += B)
        reinterpret_cast<unsigned long long *>(ctl->acc)[i] = 0ull;
    if (tid < 3)
        ctl->cursor[tid] = 0u;
    if (tid == 3) {
        ctl->out = 0u;
        ctl->bar = 0u;
    }
}

// The slot whose group this block belongs to: the last one whose blocks begin
// at or before it
__device__ __forceinline__ int run_slot(const RunArgs &A)
{
    int slot = 0, hi = A.n_slots - 1;
    while (slot < hi) {
        const int mid = (slot + hi + 1) >> 1;
        if (A.block_begin[mid] <= (int)blockIdx.x)
            slot = mid;
        else
            hi = mid - 1;
    }
    return slot;
}

// Charges: 0 one per sheet in every simulation, 1 per tracer in every one, 2
// either (a block's simulation decides)
template <int CHARGES, bool GEN>
__global__ void __launch_bounds__(B, SIC_K1_MIN_BLOCKS) k_run(const RunArgs A)
{
    const int slot = run_slot(A);
    if (CHARGES == 1 || (CHARGES == 2 && A.sims[slot].Qh != nullptr))
        run_steps<true, GEN>(A, slot);
    else
        run_steps<false, GEN>(A, slot);
}

template <int Q, bool G>
cudaError_t prep_run(size_t smem)
{
    static std::mutex mu;  // (two threads' first calls: the attribute only grows)
    static size_t done = 0;
    std::lock_guard<std::mutex> lock(mu);
    if (smem > done) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_run<Q, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        done = smem;
    }
    return cudaSuccess;
}

template <int Q, bool G>
cudaError_t run_many(const RunArgs &a, int grid, cudaStream_t s)
{
    const size_t smem = step_smem_bytes(a.nx_max, true, Q != 0);
    cudaError_t e = prep_run<Q, G>(smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(B);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_run<Q, G>, a);
    if (e == cudaSuccess)
        count_launches(1);
    return e;
}

template <int Q, bool G>
int occ_run(int nx_max)
{
    const size_t smem = step_smem_bytes(nx_max, true, Q != 0);
    if (smem > 227 * 1024 || prep_run<Q, G>(smem) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<Q, G>, B, smem) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace

cudaError_t launch_run_kernel(const RunArgs &a, int grid, int charges, bool gen, cudaStream_t s)
{
    if (charges == 0)
        return gen ? run_many<0, true>(a, grid, s) : run_many<0, false>(a, grid, s);
    if (charges == 1)
        return gen ? run_many<1, true>(a, grid, s) : run_many<1, false>(a, grid, s);
    return gen ? run_many<2, true>(a, grid, s) : run_many<2, false>(a, grid, s);
}

int run_blocks_per_sm(int nx_max, int charges, bool gen)
{
    if (charges == 0)
        return gen ? occ_run<0, true>(nx_max) : occ_run<0, false>(nx_max);
    if (charges == 1)
        return gen ? occ_run<1, true>(nx_max) : occ_run<1, false>(nx_max);
    return gen ? occ_run<2, true>(nx_max) : occ_run<2, false>(nx_max);
}

}  // namespace sic
