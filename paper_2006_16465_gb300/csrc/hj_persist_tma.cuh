// hj_persist_tma.cuh -- persistent multi-cycle kernels (hj_persist.cuh) whose
// CTAs stage subdomains with TMA and prefetch: while a CTA sweeps one work
// item in registers, the copy engine brings the next item's iterate box
// (subdomain + halo), RHS box (and 1/d box) into shared memory.
//
// Same cycle structure, barriers, reductions and stopping rules as the
// plain persistent kernels; only the staging differs (TMA boxes instead of
// predicated global loads, zero fill beyond the grid either way), so the
// iterates are identical.  Each problem has tensor maps of its two iterate
// buffers, its RHS and its 1/d in device memory (PersistMaps).
//
// Ordering: within a launch, cycle c's stores (generic proxy) are read by
// cycle c+1's copies (async proxy).  Every thread fences its stores towards
// the async proxy before the grid barrier, and the thread that issues copies
// fences again after it; the barrier orders the CTAs.  Every mbarrier wait
// is bounded: on expiry the CTA records HJ_ERR_TIMEOUT, waits (bounded) for
// its copy in flight and returns; the other CTAs then leave at the barrier.
#pragma once

#include "hj_persist.cuh"
#include "hj_tma.cuh"

namespace hj {

struct PersistMaps {
    CUtensorMap mu[3];   // iterate buffers, box (bwu, TY + 2): cycle c reads mu[c % 2] (one problem) or mu[c % 3] (many)
    CUtensorMap mf;      // right-hand side, box (bwf, TY)
    CUtensorMap md;      // per-point 1/d, box (bwf, TY); sigma only
};

__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

// One problem (one barrier per cycle, every CTA reduces all partials itself, as
// persist2d_one_kernel); items are walked with a static stride.
template <typename S, typename T, int C, int R, int NW, int H, bool EXACT, bool SIG>
__global__ void __launch_bounds__(32 * NW) persist2d_tma_one_kernel(const PersistArgs P) {
    using L = PpcLayout<S, T, C, R, NW, H, SIG, 1>;
    constexpr int TX = L::TX, TY = L::TY;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    uint64_t *bar = (uint64_t *)(smem + L::BAR_OFF);
    T *xbuf = (T *)(smem + L::XB_OFF);
    S *su = (S *)smem;
    T *sf = (T *)(smem + L::UB_AL);
    T *sd = (T *)(smem + L::UB_AL + L::FB_AL);
    const int tid = threadIdx.x;
    const int band = band_of_lane<R, H>();
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    OneState ls{-1, HJ_OK, 0, 0.0, 0.0, 0.0, 0};
    unsigned nwait = 0;   // copies waited for (mbarrier phase parity)
    const int tx = P.prob_tiles_x[0], cnt = P.nitems;
    const PersistMaps &m = P.maps[0];
    auto issue = [&](int item) {
        const int bx = item % tx, by = item / tx;
        mbar_expect_tx(bar, L::TX_BYTES);
        tma_load_2d(su, &m.mu[ls.cycle & 1], bar, bx * TX, by * TY);
        tma_load_2d(sf, &m.mf, bar, bx * TX, by * TY + 1);
        if constexpr (SIG) tma_load_2d(sd, &m.md, bar, bx * TX, by * TY + 1);
    };
    for (long long it = 0; it < P.max_iters; ++it) {
        const int parity = (int)(it & 1);
        int i = blockIdx.x;
        if (tid == 0 && i < cnt) {
            fence_proxy_async_global();
            issue(i);
        }
        for (; i < cnt; i += gridDim.x) {
            bool ok = true;
            long long spins = 0;
            while (!mbar_try_wait(bar, nwait & 1u)) {
                if (++spins > P.spin_limit) { ok = false; break; }
            }
            if (__syncthreads_or(!ok)) {
                if (tid == 0) {
                    atomicExch(P.err, HJ_ERR_TIMEOUT);
                    long long sp = 0;
                    while (!mbar_try_wait(bar, nwait & 1u) && ++sp <= P.spin_limit) {
                    }
                }
                __syncthreads();
                return;
            }
            ++nwait;
            CycArgs a = P.probs[0];
            if (ls.cycle & 1) {
                const void *t = a.uin;
                a.uin = a.uout;
                a.uout = const_cast<void *>(t);
            }
            const int x0 = 1 + (i % tx) * TX, y0 = 1 + (i / tx) * TY, yb = y0 + band * R;
            const Coef<T> kc = make_coef<T>(a);
            Tile2D<T, C, R, SIG> t;
            stage2d_smem<S, T, C, R, H, EXACT, SIG>(t, kc, su, sf, sd, L::BWU, L::BWF, band * R,
                                                    L::UB / (int)sizeof(S), L::FB / (int)sizeof(T), a.dbg);
            __syncthreads();   // every thread is done with the boxes
            if (tid == 0 && i + (int)gridDim.x < cnt) {
                fence_proxy_async_smem();
                issue(i + gridDim.x);
            }
            typename std::conditional<EXACT, double, T>::type acc;
            if (x0 + TX - 1 <= a.nx && y0 + TY - 1 <= a.ny) {
                acc = sweeps2d<T, C, R, NW, H, EXACT, SIG, true, false>(t, kc, a.k, x0, yb, a.nx, a.ny, xbuf,
                                                                        Own{0, 0, 0, 0}, a.dbg);
                store2d<S, T, C, R, H, SIG, false>(t, a, x0, yb);
            } else {
                acc = sweeps2d<T, C, R, NW, H, EXACT, SIG, true, true>(t, kc, a.k, x0, yb, a.nx, a.ny, xbuf,
                                                                       Own{0, 0, 0, 0}, a.dbg);
                store2d<S, T, C, R, H, SIG, true>(t, a, x0, yb);
            }
            const double s = cta_sum(acc);
            const size_t pi = (size_t)parity * P.nitems + i;
            if (tid == 0 && HJ_IN(a.dbg, pi, 2 * (long long)P.nitems, 50)) P.partial[pi] = s;
        }
        fence_proxy_async_global();   // this cycle's stores, before the next cycle's copies
        if ((int)blockIdx.x == P.skip_barrier_cta) return;
        if (!grid_barrier(P)) return;
        if (one_decide(P, ls, parity, P.nitems)) return;
    }
}

// ---------------------------------------------------------------------------
// Many problems: one grid barrier per cycle.
//
// What bounded the two-barrier form was latency, not sweeps: with few problems
// left a cycle took some 20 us for 3.5 us of sweeps (k = 32).  So here
//   * the decision on ||r_c|| is taken during cycle c + 1 (three iterate buffers
//     in turn keep u_c until then), as queue entries behind the cycle's items:
//     CTAs that have run out of items do the checks while others still sweep,
//     and no barrier separates reduction and retirement;
//   * a CTA's first entry of a cycle is its own number, so that it needs no
//     atomic, and no load either while the queue has not been rebuilt; further
//     entries come from the atomic head, taken two ahead so that neither the
//     atomic nor the entry's load is waited for;
//   * the queue only shrinks within a launch, so a CTA whose number lies beyond
//     its entries leaves for good, and the barrier counts those that stay;
//   * barrier words are read and written with acquire and release instead of
//     full fences;
//   * CTAs are numbered breadth-first over the SMs (cta_rank): by block index the
//     first 48 of a full launch sit on four SMs, twelve each, so that a queue of a
//     few hundred entries swept at the speed of those four (15.5 us a cycle; 8 to 9
//     with the numbering).
// The residual sums, and with them every decision and iterate, are those of the
// two-barrier kernel.  Measured (32 x 32, k = 32, binary32 inner cycles): 64
// problems of sides 64 to 512 to 1e-8 1.13 -> 0.55 s (0.65 with CTAs numbered by
// block index, twelve per SM); 8 sigma-field problems of 256 x 256 to 1e-10, forward
// and adjoint, 0.41 -> 0.16 s.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned *p, unsigned v) {
    unsigned r;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned r;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(r) : "l"(p) : "memory");
    return r;
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Rebuild the queue from the problems still active (whole CTA; the last to
// reach the barrier, while the others wait in it).
__device__ __forceinline__ void batch_queue_rebuild(const PersistArgs &P) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        int base = 0, nact = 0;
        double pts = 0.0;   // interior points: whole numbers far below 2^53
        for (int p0 = 0; p0 < P.nprob; p0 += 32) {
            const int p = p0 + lane;
            const bool act = p < P.nprob && ((volatile ProbState *)P.state + p)->done < 0;
            const int n = act ? P.prob_nitems[p] : 0;
            int x = n;   // inclusive scan over the warp
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += y;
            }
            const unsigned mask = __ballot_sync(FULL, act);
            if (p < P.nprob) P.q_off[p] = act ? base + x - n : -1;
            if (act) P.q_probs[nact + __popc(mask & ((1u << lane) - 1u))] = p;
            pts += warp_sum(act ? (double)P.prob_points[p] : 0.0);
            base += __shfl_sync(FULL, x, 31);
            nact += __popc(mask);
        }
        if (lane == 0) {
            const int gen = P.q_state->w;
            *P.q_state = make_int4(base, nact, max(1, min((int)gridDim.x, base + nact)), gen + 1);
            *P.q_points = (long long)pts;
            *P.q_changed = 0;
        }
    }
    __syncthreads();
    for (int p = 0; p < P.nprob; ++p) {
        const int off = P.q_off[p];
        if (off < 0) continue;
        const int i0 = P.prob_item0[p], n = P.prob_nitems[p], tx = P.prob_tiles_x[p];
        for (int b = threadIdx.x; b < n; b += blockDim.x)
            if (HJ_IN(P.probs[0].dbg, off + b, P.nitems, 52)) P.q_ent[off + b] = make_int4(i0 + b, p, b % tx, b / tx);
    }
}

// Grid barrier over the `alive` CTAs of the cycle.  Nothing is read in it that the
// two words do not carry: an arrival adds 1, and 2^16 if the CTA retired a problem,
// so the last to arrive knows whether to rebuild the queue; the release word's
// lowest bit tells the others whether it was rebuilt, and only then do they read
// its state into head.  False if the wait expired or a CTA recorded an error.
__device__ __forceinline__ bool batch_barrier(const PersistArgs &P, int alive, int retired, unsigned &word, int4 &head) {
    __shared__ int s_last, s_state;
    __shared__ int4 s_head;
    __syncthreads();   // the CTA's stores are done
    if (threadIdx.x == 0) {
        const unsigned mine = 1u + (retired ? 0x10000u : 0u);
        const unsigned now = atom_add_acq_rel(P.bar, mine) + mine;
        s_last = (now & 0xffffu) == (unsigned)alive ? 1 + (now >= 0x10000u) : 0;
    }
    __syncthreads();
    const unsigned next = ((word >> 1) + 1u) << 1;
    unsigned seen = next;
    int ok = 1;
    if (s_last) {
        const int changed = s_last == 2;
        if (changed) {
            batch_queue_rebuild(P);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            *P.q_head = changed ? __ldcg(&P.q_state->z) : alive;
            if (P.tlog) {
                const long long n = *P.tlog_n;
                if (n < P.tlog_cap) {
                    P.tlog[2 * n] = global_ns();
                    P.tlog[2 * n + 1] = (unsigned long long)*(volatile long long *)P.q_points;
                }
                *P.tlog_n = n + 1;
            }
            *(volatile unsigned *)P.bar = 0u;
            seen = next | (unsigned)changed;
            st_release(P.bar + 1, seen);
        }
    } else if (threadIdx.x == 0) {
        const unsigned long long t0 = global_ns();
        for (unsigned polls = 0; (seen = ld_acquire(P.bar + 1)) == word; ++polls) {
            if ((polls & 15u) == 15u) {
                if (*(volatile int *)P.err) { ok = 0; break; }
                if (global_ns() - t0 > P.timeout_ns) {
                    atomicExch(P.err, HJ_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
    }
    if (threadIdx.x == 0) {
        if (ok && (seen & 1u)) s_head = __ldcg(P.q_state);
        s_state = ok ? 1 + (int)(seen & 1u) : 0;
    }
    __syncthreads();
    const int state = s_state;
    word = next | (state == 2 ? 1u : 0u);
    if (state == 2) head = s_head;
    return state != 0;
}

// This CTA's number when the launch's CTAs are counted SM by SM, one of each in
// turn: (its place on its SM, its SM) in lexicographic order.  slot: its place;
// the per-SM counts are complete (a grid barrier lies between).  Whole CTA calls.
__device__ __forceinline__ int cta_rank(const int *sm_ctas, int sm, int slot) {
    __shared__ int s_rank;
    if (threadIdx.x < 32) {
        int r = 0;
        for (int m = threadIdx.x; m < kSmSlots; m += 32) {
            const int c = __ldcg(sm_ctas + m);
            r += min(c, slot) + (m < sm && c > slot ? 1 : 0);
        }
        r = __reduce_add_sync(FULL, r);
        if (threadIdx.x == 0) s_rank = r;
    }
    __syncthreads();
    return s_rank;
}

// Four-warp kernels with a sigma field are held to three CTAs per SM (at most
// 168 registers instead of about 220): measured 3.5 % faster on 16 1024^2
// sigma-field problems.  The others keep the compiler's choice (a minimum of 0
// CTAs leaves it as without one; an explicit 1 let the compiler take more
// registers, and the constant-sigma kernel held to three CTAs was slower).
template <typename S, typename T, int C, int R, int NW, int H, bool EXACT, bool SIG>
__global__ void __launch_bounds__(32 * NW, (NW == 4 && SIG) ? 3 : 0) persist2d_batch_kernel(const PersistArgs P) {
    using L = PpcLayout<S, T, C, R, NW, H, SIG, 1>;
    constexpr int TX = L::TX, TY = L::TY;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    uint64_t *bar = (uint64_t *)(smem + L::BAR_OFF);
    T *xbuf = (T *)(smem + L::XB_OFF);
    S *su = (S *)smem;
    T *sf = (T *)(smem + L::UB_AL);
    T *sd = (T *)(smem + L::UB_AL + L::FB_AL);
    __shared__ int s_idx;
    __shared__ int4 s_ent;
    const int tid = threadIdx.x;
    const int band = band_of_lane<R, H>();
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    unsigned nwait = 0;   // copies waited for (mbarrier phase parity)
    unsigned word = *(volatile unsigned *)(P.bar + 1);   // (moves only once every CTA has arrived)
    int4 head = make_int4(0, 0, 0, 0);
    __shared__ int s_slot;   // (every lane of a warp is on one SM, and so is its CTA)
    unsigned sm;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
    sm %= kSmSlots;
    if (tid == 0) s_slot = atomicAdd(P.sm_ctas + sm, 1);
    // the queue of the first cycle is built behind a barrier
    if (!batch_barrier(P, (int)gridDim.x, 1, word, head)) return;
    const int me = cta_rank(P.sm_ctas, (int)sm, s_slot);
    int4 first = make_int4(0, 0, 0, 0);
    int first_of = head.w - 1;   // the rebuild `first` was read from
    // entry i of the queue; debug builds check what a wrong one would send copies and
    // stores out of range with
    auto entry = [&](int i) -> int4 {
        if (!HJ_IN(P.probs[0].dbg, i, P.nitems, 51)) return make_int4(0, 0, 0, 0);
        const int4 e = __ldcg(P.q_ent + i);
        if (!HJ_IN(P.probs[0].dbg, e.x, P.nitems, 51) || !HJ_IN(P.probs[0].dbg, e.y, P.nprob, 51))
            return make_int4(0, 0, 0, 0);
        return e;
    };
    // every active problem advances once per cycle: `it` is its cycle index
    for (long long it = 0; it < P.max_iters; ++it) {
        const int cnt = head.x, alive = head.z, total = cnt + (it > 0 ? head.y : 0);
        if (head.y == 0 || me >= alive) return;
        const int parity = (int)(it & 1), bi = (int)(it % 3), bo = (int)((it + 1) % 3);
        auto issue = [&](const int4 &e) {
            const PersistMaps &m = P.maps[e.y];
            mbar_expect_tx(bar, L::TX_BYTES);
            tma_load_2d(su, &m.mu[bi], bar, e.z * TX, e.w * TY);
            tma_load_2d(sf, &m.mf, bar, e.z * TX, e.w * TY + 1);
            if constexpr (SIG) tma_load_2d(sd, &m.md, bar, e.z * TX, e.w * TY + 1);
        };
        int i = me;
        if (first_of != head.w) {
            if (i < cnt) first = entry(i);
            first_of = head.w;
        }
        int4 e = first, en = first;
        int nidx = total;   // thread 0: the entry after the current one, and its contents (en)
        if (tid == 0) {
            if (i < cnt) {
                fence_proxy_async_global();
                issue(e);
            }
            if (total > alive) {
                nidx = atomicAdd(P.q_head, 1);
                if (nidx < cnt) en = entry(nidx);
            }
        }
        while (i < cnt) {
            int after = total;   // two ahead; read after the sweeps
            if (tid == 0 && nidx < total) after = atomicAdd(P.q_head, 1);
            bool ok = true;
            long long spins = 0;
            while (!mbar_try_wait(bar, nwait & 1u)) {
                if (++spins > P.spin_limit) { ok = false; break; }
            }
            if (__syncthreads_or(!ok)) {
                if (tid == 0) {
                    atomicExch(P.err, HJ_ERR_TIMEOUT);
                    long long sp = 0;
                    while (!mbar_try_wait(bar, nwait & 1u) && ++sp <= P.spin_limit) {
                    }
                }
                __syncthreads();
                return;
            }
            ++nwait;
            const int p = e.y;
            CycArgs a = P.probs[p];
            a.uout = bo == 0 ? const_cast<void *>(a.uin) : bo == 1 ? a.uout : P.third[p];
            const int x0 = 1 + e.z * TX, y0 = 1 + e.w * TY, yb = y0 + band * R;
            const Coef<T> kc = make_coef<T>(a);
            Tile2D<T, C, R, SIG> t;
            stage2d_smem<S, T, C, R, H, EXACT, SIG>(t, kc, su, sf, sd, L::BWU, L::BWF, band * R,
                                                    L::UB / (int)sizeof(S), L::FB / (int)sizeof(T), a.dbg);
            if (tid == 0) {
                s_idx = nidx;
                s_ent = en;
            }
            __syncthreads();   // every thread is done with the boxes, and the next entry is published
            const int inext = s_idx;
            const int4 enext = s_ent;
            if (tid == 0 && inext < cnt) {
                fence_proxy_async_smem();
                issue(enext);
            }
            typename std::conditional<EXACT, double, T>::type acc;
            if (x0 + TX - 1 <= a.nx && y0 + TY - 1 <= a.ny) {
                acc = sweeps2d<T, C, R, NW, H, EXACT, SIG, true, false>(t, kc, a.k, x0, yb, a.nx, a.ny, xbuf,
                                                                        Own{0, 0, 0, 0}, a.dbg);
                store2d<S, T, C, R, H, SIG, false>(t, a, x0, yb);
            } else {
                acc = sweeps2d<T, C, R, NW, H, EXACT, SIG, true, true>(t, kc, a.k, x0, yb, a.nx, a.ny, xbuf,
                                                                       Own{0, 0, 0, 0}, a.dbg);
                store2d<S, T, C, R, H, SIG, true>(t, a, x0, yb);
            }
            const double s = cta_sum(acc);
            const size_t pi = (size_t)parity * P.nitems + e.x;
            if (tid == 0 && HJ_IN(a.dbg, pi, 2 * (long long)P.nitems, 50)) P.partial[pi] = s;
            if (tid == 0) {
                nidx = after;
                if (nidx < cnt) en = entry(nidx);
            }
            i = inext;
            e = enext;
        }
        // entries [cnt, total): the active problems' checks of the cycle before
        int retired = 0;
        if (tid < 32) {
            int next = __shfl_sync(FULL, nidx, 0);
            while (i < total) {
                retired |= retire_check(P, __ldcg(P.q_probs + (i - cnt)), parity ^ 1);
                i = next;
                if (next < total) {
                    if (tid == 0) next = atomicAdd(P.q_head, 1);
                    next = __shfl_sync(FULL, next, 0);
                }
            }
        }
        fence_proxy_async_global();   // this cycle's stores, before the next cycle's copies
        if ((int)blockIdx.x == P.skip_barrier_cta) return;
        if (!batch_barrier(P, alive, retired, word, head)) return;
    }
}

// The kernels of many problems: batches run binary32 arithmetic only (null in binary64).
template <typename S, typename T, int C, int R, int NW, int H, bool EXACT, bool SIG, bool TMA>
constexpr PersistKernel many_kernel() {
    if constexpr (std::is_same<T, double>::value) return nullptr;
    else if constexpr (TMA) return persist2d_batch_kernel<S, T, C, R, NW, H, EXACT, SIG>;
    else return persist2d_kernel<S, T, C, R, NW, H, EXACT, SIG>;
}

}  // namespace hj

#define HJ_KP2D(S, T, C, R, NW, H, EX)                                                                    \
    {2, 32 * (C) / (H), (R) * (NW) * (H), 32 * (NW), 1,                                                  \
     {hj::many_kernel<S, T, C, R, NW, H, EX, false, false>(), hj::many_kernel<S, T, C, R, NW, H, EX, true, false>()}, \
     {hj::persist2d_one_kernel<S, T, C, R, NW, H, EX, false>, hj::persist2d_one_kernel<S, T, C, R, NW, H, EX, true>}, \
     {hj::many_kernel<S, T, C, R, NW, H, EX, false, true>(), hj::many_kernel<S, T, C, R, NW, H, EX, true, true>()}, \
     {hj::persist2d_tma_one_kernel<S, T, C, R, NW, H, EX, false>,                                       \
      hj::persist2d_tma_one_kernel<S, T, C, R, NW, H, EX, true>},                                       \
     {hj::PpcLayout<S, T, C, R, NW, H, false, 1>::SMEM, hj::PpcLayout<S, T, C, R, NW, H, true, 1>::SMEM},  \
     hj::PpcLayout<S, T, C, R, NW, H, false, 1>::BWU, hj::PpcLayout<S, T, C, R, NW, H, false, 1>::BWF}
