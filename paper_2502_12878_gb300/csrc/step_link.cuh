// Linked persistent launch of the explicit sweep (Eq. 6): the resident launch
// (step_res.cuh: one block per SM, its slices' planes in shared memory for the
// whole run) without a grid barrier.  A block needs of each step only the few
// rows of other blocks that its own rows read, so every block publishes its
// rows' new values as entries that carry their step's tag, and a reader polls
// the entries of its halo until the tag is the one it waits for: one store and
// one load across the chip per step, where a barrier costs a release, an
// arrival, a poll, and only then the copy of the halo.
//
// An entry is one or two 64-bit words, each 32 bits of the value and the
// 32-bit tag, so a word is either wholly of the awaited step or not: nothing
// else has to be ordered with it.  Entries live in a ring of LINK_RING
// iterates.  A block may run ahead of its neighbours' neighbours, but not by
// more than LINK_LAG steps of the slowest: step k waits for the stop decision on
// step k - LINK_LAG, which needs every block's residual of that step.  So an entry that step k overwrites (of iterate k + 1 - LINK_RING) was
// last needed by steps that all blocks have finished, and the iterate of a run
// that stops at step k - LINK_LAG, found out LINK_LAG steps later, is still in
// the ring.  Residuals (each block's max |r| of a step) and decisions travel
// as tagged words too, between the blocks' control warps: block 0's collects,
// applies the stop rule in step order, and publishes.
//
// The same fma chain per row in support order as every launch mode, so the
// results are the same bit for bit.  Every wait is bounded.
//
// What bounds it: one hop between SMs (500 to 900 clocks from store to poll,
// by die) and a row's chain of dependent fused multiply-adds (about 110 clocks
// each in FP64) up to 40k nodes; at 90k the FP64 pipe (5.3 of 5.6 us) or, in FP32,
// the shared-memory reads of the rows.  A slice per warp where the warps suffice, so
// that inner slices - whose rows read only the block's own - start at once and
// the others as soon as the halo is there, and polling by warps without a slice.
// us per step, FP64 / FP32, against the best of the launches with a barrier: 9,801
// rows, n = 12 1.49 / 1.34 (3.15 / 2.55); 39,601, n = 30 3.5 / 1.42 (4.78 /
// 3.24); 89,401, n = 30 5.58 / 2.08 (6.75 / 3.38); 39,601, n = 56 5.84 / 2.40
// (7.5 / 3.9); 3D 12,167, n = 70 4.91 / 1.58 (6.1 / 3.0).  A first form, whose
// last warp collected residuals and decisions between its slices, took 3.05 / 2.45 at
// 9,801 rows: every block waited for block 0's collecting.
#pragma once

#include "step_res.cuh"

namespace rbffd {

// entry words
__device__ __forceinline__ void link_put(unsigned long long* x, int64_t i, double v, unsigned tag) {
    const unsigned long long b = dbits(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(x + 2 * i),
                 "l"((b & 0xffffffffull) | t), "l"((b >> 32) | t)
                 : "memory");
}
__device__ __forceinline__ bool link_get(const unsigned long long* x, int64_t i, unsigned tag,
                                         double* v) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b)
                 : "l"(x + 2 * i) : "memory");
    *v = bitsd((a & 0xffffffffull) | (b << 32));
    return (unsigned)(a >> 32) == tag && (unsigned)(b >> 32) == tag;
}
__device__ __forceinline__ void link_put(unsigned long long* x, int64_t i, float v, unsigned tag) {
    st_relaxed(x + i, (unsigned long long)__float_as_uint(v) | ((unsigned long long)tag << 32));
}
__device__ __forceinline__ bool link_get(const unsigned long long* x, int64_t i, unsigned tag,
                                         float* v) {
    const unsigned long long a = ld_relaxed(x + i);
    *v = __uint_as_float((unsigned)a);
    return (unsigned)(a >> 32) == tag;
}

// shared memory of one block: the mbarrier, weight and local-index planes, the
// rows' f (or d32), two buffers of [own rows | halo values], the halo's slots
struct LinkLayout {
    unsigned w, idx, f, v, slot, total;
};
__host__ __device__ __forceinline__ LinkLayout link_layout(int64_t nsl, int n, int wbytes,
                                                           int64_t halo) {
    LinkLayout L;
    const unsigned ent = (unsigned)(nsl * n * SLICE), rows = (unsigned)(nsl * SLICE);
    L.w = 128;
    L.idx = L.w + res_align(ent * (unsigned)wbytes);
    L.f = L.idx + res_align(ent * 2u);
    L.v = L.f + res_align(rows * (unsigned)wbytes);
    L.slot = L.v + res_align(2u * (rows + (unsigned)halo) * (unsigned)wbytes);
    L.total = L.slot + res_align((unsigned)halo * 4u);
    return L;
}

// warp max of IEEE bits (non-negative doubles): two 32-bit reductions
__device__ __forceinline__ unsigned long long link_warp_max(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

// The control warp of a block (its last) runs beside the others: it publishes
// the block's residual of each step they finish, and reads the decisions they wait
// for; block 0's also collects the residuals and decides.  The others meet at a
// named barrier of their own, so neither the collecting nor a decision on its
// way holds a step up.
struct LinkShared {
    volatile long long done;      // steps finished by the block's compute warps
    volatile long long decided;   // decisions known: steps below this one run on
    volatile long long stop;      // the step the run stopped at, -1 before
    volatile int fail;            // a wait of this block ran out
    int go[2];                    // 1: stop; by step parity, as its readers may be a step behind
                                  // the next writer
};

// one attempt to decide step q (block 0's control warp): -1 not every residual
// is there, else the stop rule's outcome, published
__device__ __forceinline__ int link_decide(const StepArgs& A, StepCtrl* c, long long q,
                                           long long k0, long long kmax, double tol, double* R0) {
    const int lane = threadIdx.x & 31;
    const unsigned tag = A.lk_epoch + (unsigned)(q - k0) + 1u;
    const unsigned long long* r = A.lk_res + (q % LINK_RING) * 2 * gridDim.x;
    unsigned long long m = 0;
    bool all = true;
    for (int b = lane; b < (int)gridDim.x; b += 32) {
        double v;
        all = link_get(r, b, tag, &v) && all;
        m = max(m, dbits(v));
    }
    if (!__all_sync(0xffffffffu, all)) return -1;
    const double R = bitsd(link_warp_max(m));
    const long long in_seg = A.lk_seg > 0 ? (q - k0) % A.lk_seg : q - k0;
    if (in_seg == 0) *R0 = R;
    int dn = stop_rule(R, *R0, in_seg, kmax, tol);
    if (dn == DONE_RUNNING && q + 1 >= kmax) dn = DONE_CAP;
    if (lane == 0) {
        st_relaxed(A.lk_dec + q % LINK_RING,
                   (unsigned long long)dn | ((unsigned long long)tag << 32));
        if (dn != DONE_RUNNING) {
            volatile StepCtrl* vc = c;
            vc->res_first = *R0;
            vc->res_last = R;
            vc->k = q + 1;
            vc->done = dn;
        }
    }
    return dn;
}

// wm [LINK_RING][nw]: the residual maxima of each step of the `used` compute
// warps that have slices
__device__ __forceinline__ void link_control(const StepArgs& A, StepCtrl* c, LinkShared& S,
                                             const unsigned long long* wm, int nw, int used,
                                             long long k0, long long kmax, long long spin,
                                             int held) {
    const int lane = threadIdx.x & 31;
    const double tol = ((volatile StepCtrl*)c)->tol;
    double R0 = 0.0;
    long long pub = k0, dec = k0;   // steps published, decisions known
    long long t0 = clock64();
    while (dec < kmax) {
        bool moved = false;
        const long long done = __shfl_sync(0xffffffffu, (long long)S.done, 0);
        if (pub < kmax && done > pub) {
            __threadfence_block();
            const unsigned long long m =
                link_warp_max(lane < used ? wm[(int)(pub % LINK_RING) * nw + lane] : 0ull);
            if (lane == 0)
                link_put(A.lk_res + (pub % LINK_RING) * 2 * gridDim.x, blockIdx.x, bitsd(m),
                         A.lk_epoch + (unsigned)(pub - k0) + 1u);
            ++pub;
            moved = true;
        }
        int dn = -1;
        if (blockIdx.x == 0) {
            if (dec < pub && held == 0) dn = link_decide(A, c, dec, k0, kmax, tol, &R0);
        } else {
            // (one address for the whole warp: the same answer in every lane)
            const unsigned long long v = ld_relaxed(A.lk_dec + dec % LINK_RING);
            const unsigned tag = A.lk_epoch + (unsigned)(dec - k0) + 1u;
            dn = __shfl_sync(0xffffffffu, (unsigned)(v >> 32) == tag ? (int)(unsigned)v : -1, 0);
        }
        if (dn >= 0) {
            if (lane == 0) {
                if (dn != DONE_RUNNING) S.stop = dec;
                S.decided = dec + 1;
            }
            if (dn != DONE_RUNNING) return;
            ++dec;
            moved = true;
        }
        const int fail = __shfl_sync(0xffffffffu, S.fail, 0);
        if (fail) return;
        const long long now = clock64();
        if (moved) t0 = now;
        if (__shfl_sync(0xffffffffu, now - t0 > spin ? 1 : 0, 0)) {
            if (lane == 0) S.fail = 1;
            return;
        }
        __syncwarp();
    }
}

// poll the entry of slot q until it is of the awaited step.  Blocks leave a run
// that stopped at different steps, as each learns of the stop at its own time, so
// the entry's owner may have left before the step that writes it.  Then this block
// is beyond the stop too and its value no longer matters: the wait also ends, not
// as a failure, when the stop is known here (the control warp polls it on its own).
template <class T>
__device__ __forceinline__ bool link_wait(const unsigned long long* x, int32_t q, unsigned tag,
                                          T* to, long long spin, const LinkShared& S) {
    T v;
    if (!link_get(x, q, tag, &v)) {
        const long long t0 = clock64();
        for (unsigned i = 1; !link_get(x, q, tag, &v); ++i)   // (the rare ends every 16 looks)
            if ((i & 15u) == 0) {
                if (S.stop >= 0) break;
                if (clock64() - t0 > spin) return false;
            }
    }
    *to = v;
    return true;
}

// barrier of the compute warps (TC threads); `bad` or-ed over them
template <int TC>
__device__ __forceinline__ bool link_sync_or(bool bad) {
    int r;
    asm volatile(
        "{ .reg .pred p, q; setp.ne.s32 p, %1, 0; barrier.cta.red.or.pred q, 1, %2, p; "
        "selp.s32 %0, 1, 0, q; }"
        : "=r"(r) : "r"(bad ? 1 : 0), "n"(TC) : "memory");
    return r != 0;
}
// MODE_POWER64: y <- dt (W_II y) with dt an exact power of two (the power
// iteration; boundary slots hold 0), max |y| in the residual's place.
template <int NN, int MODE, int TH>
__global__ void __launch_bounds__(TH, 1) link_kernel(StepArgs A, StepCtrl* c) {
    constexpr bool F64 = MODE != MODE_INNER32;
    typedef typename std::conditional<F64, double, float>::type T;
    constexpr int EW = F64 ? 2 : 1;   // words of an entry
    constexpr int NW = TH / 32 - 1, TC = 32 * NW;      // compute warps, and their threads
    extern __shared__ __align__(128) unsigned char rsm[];
    __shared__ unsigned long long s_wm[LINK_RING * NW];
    __shared__ LinkShared S;
    __shared__ long long s_k, s_max, s_spin;
    __shared__ int s_held;
    __shared__ double s_dt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t s0, s1;
    res_range(A.nslices, &s0, &s1);
    const int nsl = (int)(s1 - s0);
    const int n = NN > 0 ? NN : A.n;
    const int h0 = A.lk_off[2 * blockIdx.x];
    const int nh = A.lk_off[2 * blockIdx.x + 1];   // halo slots, the boundary's last
    const LinkLayout L = link_layout(nsl, n, (int)sizeof(T), A.lk_max);
    T* w_s = reinterpret_cast<T*>(rsm + L.w);
    uint16_t* idx_s = reinterpret_cast<uint16_t*>(rsm + L.idx);
    T* f_s = reinterpret_cast<T*>(rsm + L.f);
    T* v_s = reinterpret_cast<T*>(rsm + L.v);
    int32_t* slot_s = reinterpret_cast<int32_t*>(rsm + L.slot);
    const int r0 = (int)(s0 * SLICE), NI = (int)A.NI;
    const int rows = nsl * SLICE, vlen = rows + (int)A.lk_max;
    const int nown = max(0, min(rows, NI - r0));
    const uint32_t mbar = smem_addr(rsm);
    if (threadIdx.x == 0) {
        volatile StepCtrl* vc = c;
        s_k = vc->k;
        s_max = vc->max_steps;
        s_dt = vc->dt;
        constexpr long long dflt = SPIN_LIMIT_CYCLES;
        const long long lim = vc->spin_limit;
        s_spin = lim > 0 ? lim : dflt;
        s_held = vc->held;
        S.done = S.decided = s_k;
        S.stop = -1;
        S.fail = 0;
        S.go[0] = S.go[1] = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    // the planes: bulk copies in chunks (16-byte aligned, multiples of 16 bytes),
    // while the threads load the start iterate
    if (threadIdx.x == 0) {
        const unsigned ent = (unsigned)(nsl * n * SLICE);
        const T* wg = (F64 ? (const T*)(const void*)A.w64
                                            : (const T*)(const void*)A.w32) +
                      s0 * (int64_t)n * SLICE;
        const T* fg = (F64 ? (const T*)(const void*)A.f
                                            : (const T*)(const void*)A.d32) +
                      s0 * SLICE;
        const void* src[3] = {wg, A.lk_idx + s0 * (int64_t)n * SLICE, fg};
        const uint32_t dst[3] = {smem_addr(w_s), smem_addr(idx_s), smem_addr(f_s)};
        const unsigned bytes[3] = {ent * (unsigned)sizeof(T), ent * 2u,
                                   (unsigned)rows * (unsigned)sizeof(T)};
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar),
                     "r"(bytes[0] + bytes[1] + bytes[2]) : "memory");
        for (int q = 0; q < 3; ++q)
            for (unsigned o = 0; o < bytes[q]; o += RES_COPY_CHUNK)
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
                    "[%0], [%1], %2, [%3];" ::"r"(dst[q] + o),
                    "l"((const unsigned char*)src[q] + o), "r"(min(RES_COPY_CHUNK, bytes[q] - o)),
                    "r"(mbar)
                    : "memory");
    }
    T* u0 = F64 ? (T*)(void*)A.u0 : (T*)(void*)A.e0;
    T* u1 = F64 ? (T*)(void*)A.u1 : (T*)(void*)A.e1;
    const long long kmax = s_max, k0 = s_k, spin = s_spin;
    const T* ustart = (k0 & 1) ? u1 : u0;
    for (int i = threadIdx.x; i < nown; i += TH) v_s[(k0 & 1) * vlen + i] = ustart[r0 + i];
    for (int i = threadIdx.x; i < nh; i += TH) {
        const int32_t q = A.lk_slot[h0 + i];
        slot_s[i] = q;
        const T v = ustart[q];
        v_s[rows + i] = v;          // both buffers: boundary values stay
        v_s[vlen + rows + i] = v;
    }
    if (!mbar_wait(mbar, 0, spin)) S.fail = 1;
    __syncthreads();
    if (S.fail) {
        __syncthreads();
        if (threadIdx.x == 0) {
            atomicExch(&c->done, DONE_TIMEOUT);
            mbar_drain(mbar, 0, spin);
        }
        __syncthreads();
        return;
    }
    if (warp == NW) {
        link_control(A, c, S, s_wm, NW, min(nsl, NW), k0, kmax, spin, s_held);
        return;
    }
    int nint = 0;   // the halo's interior slots: slots ascend, boundary slots (>= NI) last
    {
        int a = 0, b = nh;
        while (a < b) {
            const int m = (a + b) >> 1;
            if (slot_s[m] < NI) a = m + 1;
            else b = m;
        }
        nint = a;
    }
    const double dt = s_dt;
    const float dt32 = (float)dt;
    const int nin = A.inner ? A.inner[blockIdx.x] : 0;   // leading slices of inner rows
    const int64_t ring = EW * A.NI;                      // words of one iterate
    unsigned long long* const X = A.lk_x;
    // a row's residual as IEEE bits of its own type (widened once per step)
    typedef typename std::conditional<F64, unsigned long long, unsigned>::type B;
    // one slice of a step: row ls * 32 + lane
    auto row = [&](int ls, const T* vc, T* vn, unsigned long long* xn, unsigned tag, B& m) {
        const int lr = ls * SLICE + lane;
        if (lr >= nown) return;
        const int eo = ls * n * SLICE + lane;
        const T acc = row_dot_far<NN, T>(w_s + eo, idx_s + eo, vc, n);
        T v;
        if constexpr (MODE == MODE_POWER64) {
            v = __dmul_rn(acc, dt);
            m = max(m, abs_bits(v));
        } else if constexpr (MODE == MODE_SWEEP64) {
            const double r = __dsub_rn(acc, f_s[lr]);
            v = __fma_rn(dt, r, vc[lr]);
            m = max(m, abs_bits(r));
        } else {
            const float r = __fadd_rn(acc, f_s[lr]);
            v = __fmaf_rn(dt32, r, vc[lr]);
            const unsigned b = __float_as_uint(r) & 0x7fffffffu;
            m = max(m, b > 0x7f800000u ? 0x7f800000u : b);   // NaN as +Inf
        }
        link_put(xn, r0 + lr, v, tag);
        vn[lr] = v;
    };
    // Slices to warps in order (inner ones lead): slice i to warp i % NW.  Warps
    // without a slice poll the halo, as many as it needs; if there is none, the
    // warps with other than inner slices do.  Those warps wait for the whole
    // halo at barrier 2 before their first such slice; inner slices wait for nothing.
    const int idle = NW - min(nsl, NW);
    const int npoll = min(idle, (nint + 31) / 32);
    const bool outer = warp < nsl && (warp >= nin || warp + (nsl - 1 - warp) / NW * NW >= nin);
    const bool polls = npoll > 0 ? warp >= nsl && warp < nsl + npoll : outer;
    // warps with an outer slice: all but those whose last slice is an inner one
    int nouter = 0;
    for (int w = 0; w < min(nsl, NW); ++w)
        nouter += w + (nsl - 1 - w) / NW * NW >= nin;
    const int pfirst = npoll > 0 ? (warp - nsl) * 32 + lane : 0;
    int pstart = pfirst, pstep = npoll * 32;
    if (npoll == 0 && outer) {   // this warp's place among the warps with outer slices
        int before = 0;
        for (int w = 0; w < warp; ++w) before += w + (nsl - 1 - w) / NW * NW >= nin;
        pstart = before * 32 + lane;
        pstep = nouter * 32;
    }
    const int hcount = 32 * (nouter + npoll);   // threads at barrier 2
    const bool checker = threadIdx.x == TC - 32;   // reads the decisions (the last warp)
    bool ended = kmax <= k0, failed = false;   // (the same in every compute thread)
    int ri = (int)(k0 % LINK_RING);
    unsigned tag = A.lk_epoch;                  // u^k's; u^{k+1}'s is tag + 1
    T* vc = v_s + (k0 & 1) * vlen;
    T* vn = v_s + ((k0 + 1) & 1) * vlen;
    const unsigned long long* xc = X + ri * ring;
    for (long long k = k0; !ended; ) {
        const int rn = ri + 1 == LINK_RING ? 0 : ri + 1;
        unsigned long long* xn = X + rn * ring;
        B m = 0;
        bool bad = false, have = k == k0;   // the start iterate's halo is there
        if constexpr (MODE == MODE_SWEEP64) {
            if (A.rec && (k - k0) % A.rec_every == 0) {
                double* to = A.rec + (k - k0) / A.rec_every * A.N;
                for (int i = threadIdx.x; i < nown; i += TC) to[A.perm[r0 + i]] = vc[i];
            }
        }
        if (npoll > 0 && polls && !have) {
            for (int i = pstart; i < nint; i += pstep)
                bad = !link_wait(xc, slot_s[i], tag, vc + rows + i, spin, S) || bad;
            asm volatile("barrier.cta.arrive 2, %0;" ::"r"(hcount) : "memory");
        }
        for (int i = warp; i < nsl; i += NW) {
            if (i >= nin && !have) {
                if (npoll == 0)
                    for (int j = pstart; j < nint; j += pstep)
                        bad = !link_wait(xc, slot_s[j], tag, vc + rows + j, spin, S) || bad;
                asm volatile("barrier.cta.sync 2, %0;" ::"r"(hcount) : "memory");
                have = true;
            }
            row(i, vc, vn, xn, tag + 1u, m);
        }
        if (warp < nsl) {
            if constexpr (F64) {
                m = link_warp_max(m);
                if (lane == 0) s_wm[ri * NW + warp] = m;
            } else {
                m = __reduce_max_sync(0xffffffffu, m);
                if (lane == 0) s_wm[ri * NW + warp] = dbits((double)__uint_as_float(m));
            }
        }
        ++k;
        if (checker) {
            // step k may run once the decision on step k - LINK_LAG is known; a
            // later one that is known already counts too
            const long long t0 = clock64();
            while (S.decided <= k - LINK_LAG && S.stop < 0 && !S.fail)
                if (clock64() - t0 > spin) {
                    bad = true;
                    break;
                }
            bad = bad || S.fail;
            S.go[k & 1] = S.stop >= 0 ? 1 : 0;
        }
        // u^k's own rows, the step's maxima and go are complete behind it
        failed = link_sync_or<TC>(bad);
        if (checker) {
            __threadfence_block();
            S.done = k;
        }
        ended = failed || S.go[k & 1];
        if (k == kmax) break;
        ri = rn;
        ++tag;
        xc = xn;
        T* t = vc;
        vc = vn;
        vn = t;
    }
    if (!ended) {   // the cap: the decisions still out, the last step's among them
        bool bad = false;
        if (checker) {
            const long long t0 = clock64();
            while (S.stop < 0 && !S.fail)
                if (clock64() - t0 > spin) {
                    bad = true;
                    break;
                }
            bad = bad || S.fail;
        }
        failed = link_sync_or<TC>(bad);
    }
    if (failed) {
        if (threadIdx.x == 0) {
            S.fail = 1;
            atomicExch(&c->done, DONE_TIMEOUT);
        }
        return;
    }
    if (kmax <= k0) return;   // no step was asked for
    // the result u^{stop + 1}: this block's rows from the ring
    const long long ks = S.stop + 1;
    const unsigned long long* xr = X + (ks % LINK_RING) * ring;
    T* uout = (ks & 1) ? u1 : u0;
    for (int i = threadIdx.x; i < nown; i += TC) {
        T v;
        link_get(xr, r0 + i, 0u, &v);
        uout[r0 + i] = v;
    }
}

}  // namespace rbffd
