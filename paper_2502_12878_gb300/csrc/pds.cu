// rbffd_nodes_pds: Poisson-disc node placement in 2D (Sec. II-C, last
// paragraph, after the method of Slak and Kosec that the paper cites).
//
// The method walks a node list first in, first out: the list starts with the
// boundary nodes (seeds); node p proposes K candidates at distance h, a fixed
// set of K directions rotated by an angle drawn for p; a candidate inside the
// domain is appended when no node in the list is closer than zeta h.
//
// Walking the list in order is a breadth-first walk by generation: the
// children of generation g are appended while generation g is walked, and
// none of them is walked before all of generation g.  So one generation can
// be processed in parallel with the same result:
//   A every candidate of the generation is tested against the nodes of all
//     earlier generations (a uniform grid with at most one node per cell);
//     those that pass take a slot (any order) and enter their cell's list;
//   C each passing candidate's conflicts of lower key - (parent's position,
//     direction j) - are collected from the lists of the cells around it;
//   D among the candidates that pass, the walk accepts, in key order, each
//     that no accepted candidate of lower key is closer to than zeta h: the
//     lexicographically first maximal independent set of the conflict graph.
//     A candidate is decided IN once all its lower-key neighbours are OUT, and
//     OUT once one of them is IN; whatever the order in which the threads
//     find that out, the set is the sequential walk's (the lowest undecided
//     key can always be decided).  The accepted ones are appended in key
//     order: they are the next generation.
// One cooperative launch walks all generations, one block per SM, with a
// counter barrier behind A, C and D.  D is one block's work on states and
// conflict lists in shared memory; the others empty the cell lists and
// compute the rotations of the nodes that the next generation may append.
//
// What bounds it: latency - about 20 dependent memory round trips and three
// barriers a generation, and the chains of the conflict graph (about 100 deep
// at any h, 2.2 conflicts a candidate).  Proximity is decided in FP32 from
// positions relative to the cells wherever that is certain (its error is below
// a ten-thousandth of zeta h), in FP64 as defined otherwise (the parent, at
// distance h, always).  Square of 218k nodes (272 generations): seven launches
// a generation 48.0 ms, this kernel 12.2; 873k nodes (530 generations) 105 and
// 41.  Of a generation's 102 kclk at 218k nodes A takes 9, C 7, the barriers 11, D 67
// (lists into shared memory 8, decisions 43, appending 10).
// Arithmetic (angles, rotations, squared distances) is a fixed sequence of
// separately rounded IEEE operations, so the node list is reproducible bit
// for bit by a sequential implementation of the same definition.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "nodegen.cuh"

namespace rbffd {

static constexpr int PDS_KMAX = 64;
static constexpr int PDS_BLOCK = 1024;
static constexpr int PDS_HITS = 64;        // conflicts a warp collects in shared memory

enum : unsigned char { PDS_UND = 0, PDS_IN = 1, PDS_OUT = 2 };

struct PdsCtrl {
    long long N;        // nodes in the list
    long long rounds;   // generations walked
    long long passes;   // most fruitless looks of a thread, summed over the generations
    unsigned long long arrivals;   // block arrivals at barriers
    int nv[2];          // slots taken by a generation's passing candidates, by its parity
    int nnz[2];         // conflict-list entries
    int err;            // 1 two nodes in one grid cell, 2 generation too large, 3 list
                        // full, 4 conflict lists too large, 6 a wait ran out
    int pad;
};

// a passing candidate: its position relative to its cell (in cells), the next
// slot of its cell's list, its key a * K + j (a: parent's place in its generation)
struct PdsCand {
    float ox, oy;
    int next, key;
};

struct PdsArgs {
    double* X;
    double* Y;
    uint8_t* B;
    double* rc;          // [maxn] cos of each node's rotation angle
    double* rs;          // [maxn] sin
    int32_t* cell;       // [G*G] node id per cell, -1 empty
    uint32_t* cpos;      // [G*G] its position in the cell (pds_q16), ~0 empty
    int32_t* chead;      // [G*G] candidate list heads, -1 empty
    PdsCand* cand;       // [capC] by slot
    double2* cxy;        // [capC] candidate positions
    int32_t* ccell;      // [capC] and grid cells
    int32_t* off;        // [capC] start of each slot's conflict list
    int32_t* adj;        // [capA] the lists: slots of lower key, -1 at the end
    uint8_t* state;      // [capC] (when shared memory is too small)
    uint32_t* pass;      // [capW] passing keys, one bit each
    // when shared memory is too small: counts before each word, accepted bits by
    // place in key order, slot of each place, place of each slot, list starts by place
    int32_t* before;     // [capW]
    uint32_t* accw;      // [capW]
    int32_t* ord;        // [capC]
    int32_t* plc;        // [capC]
    int32_t* offp;       // [capC]
    const double* ex;    // [K] fixed candidate directions
    const double* ey;
    PdsCtrl* ctrl;
    int shape, K;
    double h, cs, r2;
    double inv_cs64;     // 1 / cs
    float inv_cs;        // 1 / cs in FP32, for grid cells
    float rc2;           // (zeta h / cs)^2
    int64_t G, maxn, capF, capA, nseeds;
    int smem_bytes;
    uint64_t seed;
};

__device__ __forceinline__ bool pds_inside(int shape, double x, double y) {
    if (shape == 0) return x > 0.0 && x < 1.0 && y > 0.0 && y < 1.0;
    double dx = __dsub_rn(x, 0.5), dy = __dsub_rn(y, 0.5);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)) < 0.25;
}

__device__ __forceinline__ double pds_d2(double ax, double ay, double bx, double by) {
    double dx = __dsub_rn(ax, bx), dy = __dsub_rn(ay, by);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}

// Grid cell of a point in [0, 1]^2, in FP32.  The grid only accelerates the
// proximity tests (every decision is that of the exact FP64 squared
// distances), so any cell map keeping two properties gives the same node list:
// at most one node per cell and every node within zeta h of a point inside the
// 5 x 5 cells around the point's cell.  With cells of side 0.99 zeta h / sqrt 2,
// FP32 rounding (below 1e-7 in the unit square, h >= 5e-5) moves a point by
// far less than the 1 % margin on both.  One FP64 division per axis would
// cost more than the rest of a candidate's work on this GPU's FP64 pipe.
__device__ __forceinline__ void pds_cell_xy(const PdsArgs& A, double x, double y, int* gx,
                                            int* gy) {
    const int a = (int)__fmul_rn(__double2float_rn(x), A.inv_cs);
    const int b = (int)__fmul_rn(__double2float_rn(y), A.inv_cs);
    const int G = (int)A.G;
    *gx = a < 0 ? 0 : (a >= G ? G - 1 : a);
    *gy = b < 0 ? 0 : (b >= G ? G - 1 : b);
}

// position relative to the cell, in cells: within 1e-6 of the true one, and
// in [-0.01, 1.01] (the FP32 cell map moves a point by at most 0.004 cells)
__device__ __forceinline__ float pds_rel(const PdsArgs& A, double x, int g) {
    return (float)__dmul_rn(__fma_rn(-(double)g, A.cs, x), A.inv_cs64);
}

// a node's relative position in 16 bits an axis (steps of 2^-15 cells from
// -1/4, so within 1.6e-5 cells; never all ones)
__device__ __forceinline__ unsigned pds_q16(float o) {
    return (unsigned)fminf(fmaxf((o + 0.25f) * 32768.f, 0.f), 65535.f);
}
__device__ __forceinline__ float pds_o16(unsigned q) {
    return ((float)(int)(q & 0xffffu) + 0.5f) * (1.f / 32768.f) - 0.25f;
}
__device__ __forceinline__ bool pds_put_node(const PdsArgs& A, int64_t id, int64_t c, float ox,
                                             float oy) {
    A.cpos[c] = (pds_q16(ox) << 16) | pds_q16(oy);
    return atomicCAS(&A.cell[c], -1, (int32_t)id) == -1;
}

// seeds: the boundary grid points of the square in row-major order, or the
// disk's boundary nodes at angles 2 pi k / Nb
__global__ void pds_seeds(PdsArgs A, int Kg, int64_t nb) {
    const double two_pi = 6.283185307179586;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nb;
         s += (int64_t)gridDim.x * blockDim.x) {
        double x, y;
        if (A.shape == 0) {
            int64_t i, j;
            const int64_t first = (int64_t)Kg + 1, mid = 2 * ((int64_t)Kg - 1);
            if (s < first) {
                i = 0;
                j = s;
            } else if (s < first + mid) {
                int64_t r = s - first;
                i = 1 + r / 2;
                j = (r & 1) ? Kg : 0;
            } else {
                i = Kg;
                j = s - first - mid;
            }
            x = __dmul_rn((double)i, A.h);
            y = __dmul_rn((double)j, A.h);
        } else {
            double a = __ddiv_rn(__dmul_rn(two_pi, (double)s), (double)nb);
            double ux, uy;
            unit_dir(a, &ux, &uy);
            x = __dadd_rn(0.5, __dmul_rn(0.5, ux));
            y = __dadd_rn(0.5, __dmul_rn(0.5, uy));
        }
        A.X[s] = x;
        A.Y[s] = y;
        A.B[s] = 1;
        int gx, gy;
        pds_cell_xy(A, x, y, &gx, &gy);
        if (!pds_put_node(A, s, gx * A.G + gy, pds_rel(A, x, gx), pds_rel(A, y, gy)))
            atomicExch(&A.ctrl->err, 1);
        unit_dir(__dmul_rn(two_pi, unit_draw(A.seed, (uint64_t)s)), &A.rc[s], &A.rs[s]);
    }
}

// the fixed directions e_j at angles 2 pi j / K
__global__ void pds_dirs(int K, double* ex, double* ey) {
    const double two_pi = 6.283185307179586;
    int j = threadIdx.x;
    if (j < K) unit_dir(__ddiv_rn(__dmul_rn(two_pi, (double)j), (double)K), &ex[j], &ey[j]);
}

// exclusive scan of one value per thread over a PDS_BLOCK-thread block;
// returns the thread's offset and sets *total
__device__ int block_excl_scan(int v, int* total) {
    __shared__ int ws[PDS_BLOCK / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int t = lane < PDS_BLOCK / 32 ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < PDS_BLOCK / 32) ws[lane] = t;
    }
    __syncthreads();
    const int before = (wid ? ws[wid - 1] : 0) + x - v;
    *total = ws[PDS_BLOCK / 32 - 1];
    __syncthreads();
    return before;
}

// grid barrier: every block's arrival is a release, every wait an acquire
// (bounded by the clock; false in every thread when it gave up or err is set)
static constexpr long long PDS_SPIN = 4000000000LL;   // ~2 s

__device__ __forceinline__ bool pds_barrier(PdsCtrl* c, unsigned long long* target) {
    __syncthreads();
    *target += gridDim.x;
    int ok = 1;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&c->arrivals) : "memory");
        const long long t0 = clock64();
        unsigned long long v;
        for (;;) {
            asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(&c->arrivals) : "memory");
            if (v >= *target) break;
            // a block that saw an error may not come
            if (*(volatile int*)&c->err) break;
            if (clock64() - t0 > PDS_SPIN) {
                atomicCAS(&c->err, 0, 6);
                break;
            }
        }
        if (*(volatile int*)&c->err) ok = 0;
    }
    return __syncthreads_and(ok) != 0;
}

// A: the candidates of nodes [lo, hi), one per thread
__device__ __forceinline__ void pds_generate(const PdsArgs& A, long long lo, long long hi, int par,
                                             const double* ex, const double* ey) {
    const long long total = (hi - lo) * A.K;
    const int lane = threadIdx.x & 31;
    const int G = (int)A.G;
    const float sure = A.rc2 * (1.f - 1e-4f), maybe = A.rc2 * (1.f + 1e-4f);
    // whole warps, spread over the blocks first: warp w of block b starts at
    // (w * gridDim + b) * 32
    const long long stride = (long long)gridDim.x * PDS_BLOCK;
    for (long long e0 = ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32; e0 < total;
         e0 += stride) {
        const long long e = e0 + lane;
        bool ok = false;
        double x = 0.0, y = 0.0;
        int gx = 0, gy = 0;
        float ox = 0.f, oy = 0.f;
        if (e < total) {
            const int a = (int)((unsigned)e / (unsigned)A.K);
            const int j = (int)e - a * A.K;
            const long long p = lo + a;
            const double c = A.rc[p], s = A.rs[p];
            const double ux = __dsub_rn(__dmul_rn(c, ex[j]), __dmul_rn(s, ey[j]));
            const double uy = __dadd_rn(__dmul_rn(s, ex[j]), __dmul_rn(c, ey[j]));
            x = __dadd_rn(A.X[p], __dmul_rn(A.h, ux));
            y = __dadd_rn(A.Y[p], __dmul_rn(A.h, uy));
            ok = pds_inside(A.shape, x, y);
        }
        if (ok) {
            pds_cell_xy(A, x, y, &gx, &gy);
            ox = pds_rel(A, x, gx);
            oy = pds_rel(A, y, gy);
            // the 5 x 5 cells' entries: independent loads
            uint32_t q[25];
#pragma unroll
            for (int l = 0; l < 25; ++l) {
                const int cx = gx - 2 + l / 5, cy = gy - 2 + l % 5;
                q[l] = cx >= 0 && cx < G && cy >= 0 && cy < G
                           ? A.cpos[(int64_t)cx * A.G + cy]
                           : ~0u;
            }
            unsigned open = 0;   // cells whose node FP32 cannot decide
#pragma unroll
            for (int l = 0; l < 25; ++l) {
                const float dx = (float)(l / 5 - 2) + pds_o16(q[l] >> 16) - ox;
                const float dy = (float)(l % 5 - 2) + pds_o16(q[l]) - oy;
                const float d2 = dx * dx + dy * dy;
                if (q[l] != ~0u) {
                    if (d2 < sure) ok = false;
                    else if (d2 < maybe) open |= 1u << l;
                }
            }
            while (ok && open) {
                const int l = __ffs(open) - 1;
                open &= open - 1;
                const int64_t cl = (int64_t)(gx - 2 + l / 5) * A.G + (gy - 2 + l % 5);
                const int64_t id = A.cell[cl];
                if (pds_d2(x, y, A.X[id], A.Y[id]) < A.r2) ok = false;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) A.pass[e0 / 32] = m;
        if (m) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&A.ctrl->nv[par], __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (ok) {
                const int q = base + __popc(m & ((1u << lane) - 1u));
                const int64_t cl = (int64_t)gx * A.G + gy;
                PdsCand r;
                r.ox = ox;
                r.oy = oy;
                r.next = atomicExch(&A.chead[cl], q);
                r.key = (int)e;
                A.cand[q] = r;
                A.cxy[q] = make_double2(x, y);
                A.ccell[q] = (int32_t)cl;
            }
        }
    }
}

// C: the lower-key conflicts of each slot, one warp per slot: lane l < 25
// walks the list of cell l of the 5 x 5
__device__ __forceinline__ void pds_conflicts(const PdsArgs& A, int nv, int par, int32_t* hits) {
    const int lane = threadIdx.x & 31;
    const int G = (int)A.G;
    const unsigned below = (1u << lane) - 1u;
    const float sure = A.rc2 * (1.f - 1e-5f), maybe = A.rc2 * (1.f + 1e-5f);
    const int dcx = lane / 5 - 2, dcy = lane % 5 - 2;
    for (int q = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; q < nv;
         q += gridDim.x * (PDS_BLOCK / 32)) {
        const PdsCand me = A.cand[q];
        const int cl = A.ccell[q];
        const int cx = cl / G + dcx, cy = cl % G + dcy;
        const int head = lane < 25 && cx >= 0 && cx < G && cy >= 0 && cy < G
                             ? A.chead[(int64_t)cx * A.G + cy]
                             : -1;
        int base = 0, cnt = 0;
        // first walk: count, and keep the first PDS_HITS; a second one writes
        // straight to the list when there are more
        for (int walk = 0; walk < 2; ++walk) {
            int w = head;
            cnt = 0;
            while (__any_sync(0xffffffffu, w >= 0)) {
                bool hit = false;
                int next = -1;
                if (w >= 0) {
                    const PdsCand o = A.cand[w];
                    next = o.next;
                    if (o.key < me.key) {
                        const float dx = (float)dcx + o.ox - me.ox, dy = (float)dcy + o.oy - me.oy;
                        const float d2 = dx * dx + dy * dy;
                        hit = d2 < sure;
                        if (!hit && d2 < maybe) {
                            const double2 a = A.cxy[q], b = A.cxy[w];
                            hit = pds_d2(a.x, a.y, b.x, b.y) < A.r2;
                        }
                    }
                }
                const unsigned m = __ballot_sync(0xffffffffu, hit);
                if (hit) {
                    const int at = cnt + __popc(m & below);
                    if (walk) A.adj[base + at] = w;
                    else if (at < PDS_HITS) hits[at] = w;
                }
                cnt += __popc(m);
                w = next;
            }
            __syncwarp();
            if (walk) break;
            if (lane == 0) {
                base = atomicAdd(&A.ctrl->nnz[par], cnt + 1);
                if ((long long)base + cnt + 1 > A.capA || base < 0) {
                    atomicExch(&A.ctrl->err, 4);
                    base = -1;
                }
            }
            base = __shfl_sync(0xffffffffu, base, 0);
            if (base < 0) break;
            if (lane == 0) {
                A.off[q] = base;
                A.adj[base + cnt] = -1;
            }
            if (cnt <= PDS_HITS) {
                for (int i = lane; i < cnt; i += 32) A.adj[base + i] = hits[i];
                break;
            }
        }
        __syncwarp();
    }
}

// D: decide every candidate, by place p in key order: warp w takes the 32
// candidates of chunk c = w, w + 32, ..., a lane each.  A lane's conflicts
// inside the chunk are a bit mask, settled by ballots; the others (of lower
// chunks) are looked at four at a time in their states.  No barrier: conflicts
// have lower keys, so the lowest undecided candidate is always one that a warp
// is at.  At 218k nodes (5,400 candidates a generation, chains of about 100
// conflicts) 43 kclk a generation; with every conflict looked at in shared memory, one
// at a time, 137; slots in no particular order, several a thread, each waiting
// for one conflict, 141; 8 and 16 deciding warps 58 and 45.
// accw[c]: the accepted ones of chunk c.  Bounded by the clock.
template <class Index, Index END>
__device__ __forceinline__ void pds_decide(volatile uint8_t* st, const int32_t* off,
                                           const Index* adj, int nv, uint32_t* accw, int* err,
                                           int* looks_out) {
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const long long t0 = clock64();
    int looks = 0;
    for (int c = threadIdx.x >> 5; 32 * c < nv; c += PDS_BLOCK / 32) {
        const int p = 32 * c + lane;
        bool open = p < nv;
        unsigned inside = 0;             // conflicts of this chunk
        Index e[4] = {END, END, END, END};   // conflicts of lower chunks, four at a time
        int k = open ? off[p] : 0;       // the list's next entry
        bool more = open;                // entries are left in the list
        unsigned und = __ballot_sync(FULL, open), acc = 0;
        while (und) {
            bool hit = false, blocked = false;
            if (more && e[0] == END && e[1] == END && e[2] == END && e[3] == END) {
                int have = 0;
                for (;;) {
                    const Index x = adj[k];
                    if (x == END) {
                        more = false;
                        break;
                    }
                    ++k;
                    if ((int)(x >> 5) == c) {
                        inside |= 1u << (x & 31);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (have == i) e[i] = x;
                        if (++have == 4) break;
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (e[i] != END) {
                    const unsigned char sw = st[e[i]];
                    hit = hit || sw == PDS_IN;
                    blocked = blocked || sw == PDS_UND;
                    if (sw == PDS_OUT) e[i] = END;
                }
            blocked = blocked || more;
            // settle what the chunk itself decides now
            unsigned news = 0;
            for (;;) {
                const bool out = open && (hit || (inside & acc) != 0);
                const bool in = open && !out && !blocked && (inside & und) == 0;
                const unsigned mi = __ballot_sync(FULL, in);
                const unsigned mo = __ballot_sync(FULL, out);
                if (!(mi | mo)) break;
                acc |= mi;
                und &= ~(mi | mo);
                news |= mi | mo;
                if (in || out) open = false;
            }
            if ((news >> lane) & 1u) st[p] = (acc >> lane) & 1u ? PDS_IN : PDS_OUT;
            // (one lane's clock for the warp: its lanes leave together or not at all)
            if ((++looks & 1023) == 0 &&
                __shfl_sync(FULL, clock64() - t0 > PDS_SPIN ? 1 : 0, 0)) {
                if (lane == 0) atomicCAS(err, 0, 6);
                break;
            }
        }
        if (lane == 0) accw[c] = acc;
    }
    atomicMax(looks_out, looks);
}

// D, block 0: decide, then append the accepted candidates in key order
template <class Index, Index END>
__device__ __forceinline__ void pds_append_in(const PdsArgs& A, long long hi, int nv, int nnz,
                                              int words, int32_t* before, uint32_t* accw,
                                              volatile uint8_t* st, Index* ord, Index* plc,
                                              int32_t* off, Index* adj, int* looks) {
    const int t = threadIdx.x, chunks = (nv + 31) / 32;
    // places of the passing candidates in key order
    const int per = (words + PDS_BLOCK - 1) / PDS_BLOCK;
    const int w0 = min(words, t * per), w1 = min(words, w0 + per);
    int cnt = 0;
    for (int w = w0; w < w1; ++w) cnt += __popc(A.pass[w]);
    int all;
    int pos = block_excl_scan(cnt, &all);
    for (int w = w0; w < w1; ++w) {
        before[w] = pos;
        pos += __popc(A.pass[w]);
    }
    __syncthreads();
    for (int q = t; q < nv; q += PDS_BLOCK) {
        const unsigned k = (unsigned)A.cand[q].key;
        const int p = before[k >> 5] + __popc(A.pass[k >> 5] & ((1u << (k & 31)) - 1u));
        st[q] = PDS_UND;
        plc[q] = (Index)p;
        ord[p] = (Index)q;
        off[p] = A.off[q];
    }
    __syncthreads();
    // the lists' slots become places (in global memory: in place)
#pragma unroll 4
    for (int i = t; i < nnz; i += PDS_BLOCK) {
        const int w = A.adj[i];
        adj[i] = w < 0 ? END : plc[w];
    }
    __syncthreads();
    pds_decide<Index, END>(st, off, adj, nv, accw, &A.ctrl->err, looks);
    __syncthreads();
    // accepted ones before each chunk of 32 places
    const int cper = (chunks + PDS_BLOCK - 1) / PDS_BLOCK;
    const int c0 = min(chunks, t * cper), c1 = min(chunks, c0 + cper);
    cnt = 0;
    for (int c = c0; c < c1; ++c) cnt += __popc(accw[c]);
    int nacc;
    pos = block_excl_scan(cnt, &nacc);
    for (int c = c0; c < c1; ++c) {
        before[c] = pos;
        pos += __popc(accw[c]);
    }
    __syncthreads();
    for (int p = t; p < nv; p += PDS_BLOCK) {
        const uint32_t m = accw[p >> 5];
        if (!((m >> (p & 31)) & 1u)) continue;
        const long long id = hi + before[p >> 5] + __popc(m & ((1u << (p & 31)) - 1u));
        if (id >= A.maxn) {
            atomicExch(&A.ctrl->err, 3);
            continue;
        }
        const int q = ord[p];
        const PdsCand me = A.cand[q];
        const double2 x = A.cxy[q];
        A.X[id] = x.x;
        A.Y[id] = x.y;
        A.B[id] = 0;
        if (!pds_put_node(A, id, A.ccell[q], me.ox, me.oy)) atomicExch(&A.ctrl->err, 1);
    }
    if (t == 0) {
        A.ctrl->N = hi + nacc;
        A.ctrl->rounds += 1;
    }
}

__device__ __forceinline__ void pds_append(const PdsArgs& A, long long lo, long long hi, int nv,
                                           int nnz, unsigned char* smem) {
    __shared__ int s_looks;
    const int t = threadIdx.x;
    if (t == 0) s_looks = 0;   // (a block barrier follows before its first use)
    const int words = (int)(((hi - lo) * A.K + 31) / 32), chunks = (nv + 31) / 32;
    // counts before each key word (later: before each chunk), accepted bits by
    // place, states, slot of each place, place of each slot, list starts by place
    // and conflict lists: all in shared memory, lists and slots in 16 bits (up to
    // about 13,000 candidates: squares of h >= 1/1100), or all in global memory
    auto up = [](long long b) { return (b + 15) / 16 * 16; };
    const long long o_accw = up(4LL * max(words, chunks)), o_st = o_accw + up(4LL * chunks),
                    o_ord = o_st + up(nv), o_plc = o_ord + up(2LL * nv),
                    o_off = o_plc + up(2LL * nv), o_adj = o_off + up(4LL * nv);
    const bool in_smem = nv < 65535 && o_adj + 2LL * nnz <= A.smem_bytes;
    if (in_smem)
        pds_append_in<uint16_t, (uint16_t)0xffff>(
            A, hi, nv, nnz, words, reinterpret_cast<int32_t*>(smem),
            reinterpret_cast<uint32_t*>(smem + o_accw), smem + o_st,
            reinterpret_cast<uint16_t*>(smem + o_ord), reinterpret_cast<uint16_t*>(smem + o_plc),
            reinterpret_cast<int32_t*>(smem + o_off), reinterpret_cast<uint16_t*>(smem + o_adj),
            &s_looks);
    else
        pds_append_in<int32_t, -1>(A, hi, nv, nnz, words, A.before, A.accw, A.state, A.ord, A.plc,
                                   A.offp, A.adj, &s_looks);
    if (t == 0) A.ctrl->passes += s_looks;
}

// the walk: all generations
__global__ void __launch_bounds__(PDS_BLOCK, 1) pds_walk(PdsArgs A) {
    extern __shared__ __align__(16) unsigned char pds_smem[];
    __shared__ double s_ex[PDS_KMAX], s_ey[PDS_KMAX];
    __shared__ int32_t s_hits[PDS_BLOCK / 32][PDS_HITS];
    const double two_pi = 6.283185307179586;
    const int t = threadIdx.x;
    if (t < A.K) {
        s_ex[t] = A.ex[t];
        s_ey[t] = A.ey[t];
    }
    __syncthreads();
    unsigned long long target = 0;
    long long lo = 0, hi = A.nseeds;
    long long turned = A.nseeds;   // nodes whose rotation is there (same in every block)
    // each generation appends at least one node until the walk ends, so there
    // are at most maxn of them
    for (long long g = 0; g < A.maxn && hi > lo; ++g) {
        const int par = (int)(g & 1);
        if (hi - lo > A.capF || (hi - lo) * A.K > 0x7fffffffLL) {
            if (blockIdx.x == 0 && t == 0) atomicExch(&A.ctrl->err, 2);
            return;   // in every block: lo and hi are the same everywhere
        }
        pds_generate(A, lo, hi, par, s_ex, s_ey);
        if (!pds_barrier(A.ctrl, &target)) return;
        const int nv = *(volatile int*)&A.ctrl->nv[par];
        pds_conflicts(A, nv, par, s_hits[t >> 5]);
        if (!pds_barrier(A.ctrl, &target)) return;
        if (blockIdx.x == 0) {
            if (t == 0) {   // the next generation's counters (read last before this barrier)
                A.ctrl->nv[par ^ 1] = 0;
                A.ctrl->nnz[par ^ 1] = 0;
            }
            pds_append(A, lo, hi, nv, *(volatile int*)&A.ctrl->nnz[par], pds_smem);
        }
        if (blockIdx.x > 0 || gridDim.x == 1) {
            const int b = gridDim.x == 1 ? 0 : blockIdx.x - 1, nb = gridDim.x == 1 ? 1 : gridDim.x - 1;
            // empty the lists; the rotations of the ids this generation may append
            for (int q = b * PDS_BLOCK + t; q < nv; q += nb * PDS_BLOCK)
                A.chead[A.ccell[q]] = -1;
            const long long end = min((long long)A.maxn, hi + nv);
            for (long long id0 = turned + ((long long)(t >> 5) * nb + b) * 32; id0 < end;
                 id0 += (long long)nb * PDS_BLOCK) {
                const long long id = id0 + (t & 31);
                if (id < end)
                    unit_dir(__dmul_rn(two_pi, unit_draw(A.seed, (uint64_t)id)), &A.rc[id],
                             &A.rs[id]);
            }
        }
        turned = max(turned, min((long long)A.maxn, hi + nv));
        if (!pds_barrier(A.ctrl, &target)) return;
        lo = hi;
        hi = *(volatile long long*)&A.ctrl->N;
    }
}

__global__ void pds_copy_out(const PdsArgs A, int64_t N, double* xyz, uint8_t* is_bnd,
                             int64_t cap) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        xyz[i] = A.X[i];
        xyz[cap + i] = A.Y[i];
        is_bnd[i] = A.B[i];
    }
}

static double pds_cell_side(double zeta, double h) {
    return (0.99 * (zeta * h)) / 1.4142135623730951;
}

// cells per axis over [0, 1] (one spare column for FP32 rounding at x = 1)
static int64_t pds_cells_per_axis(int Kg, double zeta) {
    return (int64_t)(1.0 / pds_cell_side(zeta, 1.0 / (double)Kg)) + 2;
}

// one attempt with room for generations of at most capF nodes; returns
// RBFFD_OK, or RBFFD_ERR_CAPACITY with *grow set when a generation was larger
static int pds_run(int shape, int Kg, int K, double zeta, uint64_t seed, int64_t capF,
                   int64_t capA, double* xyz, uint8_t* is_bnd, int64_t cap, int64_t* h_n,
                   int64_t* h_rounds, int* grow, cudaStream_t s) {
    *grow = 0;
    const double h = 1.0 / (double)Kg;
    const int64_t G = pds_cells_per_axis(Kg, zeta);
    const int64_t maxn = G * G;
    const int64_t capC = capF * K;
    const double t = zeta * h;
    PdsArgs A;
    A.shape = shape;
    A.K = K;
    A.h = h;
    A.cs = pds_cell_side(zeta, h);
    A.inv_cs = (float)(1.0 / A.cs);
    A.r2 = t * t;
    A.G = G;
    A.maxn = maxn;
    A.capF = capF;
    A.capA = capA;
    A.seed = seed;
    A.inv_cs64 = 1.0 / A.cs;
    A.rc2 = (float)((t / A.cs) * (t / A.cs));
    const int64_t capW = (capC + 31) / 32;
    size_t used = 0;
    auto take = [&](size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t oX = take(8 * maxn), oY = take(8 * maxn), oB = take(maxn), orc = take(8 * maxn),
                 ors = take(8 * maxn), ocell = take(4 * maxn), opos = take(4 * maxn), ohead = take(4 * maxn),
                 ocand = take(sizeof(PdsCand) * capC), ocxy = take(16 * capC),
                 occell = take(4 * capC), ooff = take(4 * capC), oadj = take(4 * capA),
                 ost = take(capC), opa = take(4 * capW), obe = take(4 * capW),
                 oac = take(4 * capW), oor = take(4 * capC), opl = take(4 * capC),
                 oof = take(4 * capC),
                 odir = take(16 * PDS_KMAX), octl = take(sizeof(PdsCtrl));
    Scratch mem;
    RBFFD_CHECK_CUDA(mem.alloc(used, s));
    char* base = mem.as<char>();
    A.X = (double*)(base + oX);
    A.Y = (double*)(base + oY);
    A.B = (uint8_t*)(base + oB);
    A.rc = (double*)(base + orc);
    A.rs = (double*)(base + ors);
    A.cell = (int32_t*)(base + ocell);
    A.cpos = (uint32_t*)(base + opos);
    A.chead = (int32_t*)(base + ohead);
    A.cand = (PdsCand*)(base + ocand);
    A.cxy = (double2*)(base + ocxy);
    A.ccell = (int32_t*)(base + occell);
    A.off = (int32_t*)(base + ooff);
    A.adj = (int32_t*)(base + oadj);
    A.state = (uint8_t*)(base + ost);
    A.pass = (uint32_t*)(base + opa);
    A.before = (int32_t*)(base + obe);
    A.accw = (uint32_t*)(base + oac);
    A.ord = (int32_t*)(base + oor);
    A.plc = (int32_t*)(base + opl);
    A.offp = (int32_t*)(base + oof);
    double* dirs = (double*)(base + odir);
    A.ex = dirs;
    A.ey = dirs + PDS_KMAX;
    A.ctrl = (PdsCtrl*)(base + octl);
    RBFFD_CHECK_CUDA(cudaMemsetAsync(A.cell, 0xff, 4 * maxn, s));
    RBFFD_CHECK_CUDA(cudaMemsetAsync(A.cpos, 0xff, 4 * maxn, s));
    RBFFD_CHECK_CUDA(cudaMemsetAsync(A.chead, 0xff, 4 * maxn, s));
    const int64_t nb = shape == 0 ? 4 * (int64_t)Kg
                                  : (int64_t)floor((6.283185307179586 * 0.5) / h + 0.5);
    A.nseeds = nb;
    PdsCtrl hc;
    memset(&hc, 0, sizeof(hc));
    hc.N = nb;
    RBFFD_CHECK_CUDA(cudaMemcpyAsync(A.ctrl, &hc, sizeof(hc), cudaMemcpyHostToDevice, s));
    pds_dirs<<<1, PDS_KMAX, 0, s>>>(K, dirs, dirs + PDS_KMAX);
    pds_seeds<<<(unsigned)((nb + 255) / 256), 256, 0, s>>>(A, Kg, nb);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    const unsigned grid = (unsigned)device_sm_count() * 4;
    A.smem_bytes = 200 * 1024;   // states and conflict lists of the deciding block
    RBFFD_CHECK_CUDA(cudaFuncSetAttribute((const void*)pds_walk,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          A.smem_bytes));
    int per_sm = 0;
    RBFFD_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, (const void*)pds_walk, PDS_BLOCK, A.smem_bytes));
    void* args[] = {(void*)&A};
    RBFFD_CHECK_CUDA(cudaLaunchCooperativeKernel((const void*)pds_walk,
                                                 dim3(device_sm_count() * std::max(1, per_sm)),
                                                 dim3(PDS_BLOCK), args, A.smem_bytes, s));
    RBFFD_CHECK_CUDA(cudaMemcpyAsync(&hc, A.ctrl, sizeof(hc), cudaMemcpyDeviceToHost, s));
    RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
    if (hc.err == 2 || hc.err == 4) {
        *grow = hc.err;
        return RBFFD_ERR_CAPACITY;
    }
    if (hc.err == 6) {
        set_error("rbffd_nodes_pds: a wait between the walk's blocks ran out");
        return RBFFD_ERR_TIMEOUT;
    }
    if (hc.err) {
        set_error("rbffd_nodes_pds: internal error %d (grid cell collision or list full)",
                  hc.err);
        return RBFFD_ERR_CUDA;
    }
    *h_n = hc.N;
    if (h_rounds) {
        h_rounds[0] = hc.rounds;
        h_rounds[1] = hc.passes;
    }
    if (hc.N > cap) {
        set_error("rbffd_nodes_pds: %lld nodes, capacity %lld", (long long)hc.N,
                  (long long)cap);
        return RBFFD_ERR_CAPACITY;
    }
    pds_copy_out<<<grid, 256, 0, s>>>(A, hc.N, xyz, is_bnd, cap);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
    return RBFFD_OK;
}

// the 3D walk (pds3.cu)
int pds3_run(int Kg, int K, double zeta, uint64_t seed, double* xyz, uint8_t* is_bnd,
             int64_t cap, int64_t* h_n, int64_t* h_rounds, cudaStream_t s);
int64_t pds3_node_bound(int Kg, double zeta);

}  // namespace rbffd

using namespace rbffd;

extern "C" int rbffd_nodes_pds_cap(int d, int Kg, double zeta, int64_t* h_cap) {
    clear_error();
    RBFFD_ARG(h_cap, "rbffd_nodes_pds_cap: NULL argument");
    RBFFD_ARG(d == 2 || d == 3, "rbffd_nodes_pds_cap: d must be 2 or 3");
    RBFFD_ARG(Kg >= 2 && Kg <= (d == 2 ? 20000 : 1000) && zeta > 0.0 && zeta <= 1.0,
              "rbffd_nodes_pds_cap: bad Kg / zeta");
    if (d == 3) {
        *h_cap = pds3_node_bound(Kg, zeta);
        return RBFFD_OK;
    }
    const int64_t G = pds_cells_per_axis(Kg, zeta);
    *h_cap = G * G;
    return RBFFD_OK;
}

extern "C" int rbffd_nodes_pds(int d, int shape, int Kg, int K, double zeta, uint64_t seed,
                               double* xyz, uint8_t* is_bnd, int64_t cap, int64_t* h_n_out,
                               int64_t* h_rounds, void* stream) {
    clear_error();
    RBFFD_ARG(d == 2 || d == 3, "rbffd_nodes_pds: d must be 2 or 3");
    RBFFD_ARG(shape == 0 || (shape == 1 && d == 2),
              "rbffd_nodes_pds: shape must be 0 (square / cube) or 1 (disk, d = 2)");
    RBFFD_ARG(Kg >= 2 && Kg <= (d == 2 ? 20000 : 1000),
              "rbffd_nodes_pds: Kg must be in [2, 20000] (d = 2) or [2, 1000] (d = 3)");
    RBFFD_ARG(K >= 1 && K <= (d == 2 ? PDS_KMAX : 256),
              "rbffd_nodes_pds: K must be in [1, 64] (d = 2) or [1, 256] (d = 3)");
    RBFFD_ARG(zeta > 0.0 && zeta <= 1.0, "rbffd_nodes_pds: zeta must be in (0, 1]");
    RBFFD_ARG(h_n_out && (cap == 0 || (xyz && is_bnd)), "rbffd_nodes_pds: NULL argument");
    cudaStream_t s = as_stream(stream);
    if (d == 3) return pds3_run(Kg, K, zeta, seed, xyz, is_bnd, cap, h_n_out, h_rounds, s);
    const int64_t G = pds_cells_per_axis(Kg, zeta);
    int64_t capF = std::min<int64_t>(G * G, 64 * G + 4096);
    int64_t capA = 8 * capF * K;
    for (int attempt = 0; attempt < 8; ++attempt) {
        int grow = 0;
        int st = pds_run(shape, Kg, K, zeta, seed, capF, capA, xyz, is_bnd, cap, h_n_out,
                         h_rounds, &grow, s);
        if (!grow) return st;
        if (grow == 2) capF = std::min<int64_t>(G * G, capF * 4);
        capA *= 4;
        if (capA > (int64_t(1) << 31) - 1) break;
    }
    set_error("rbffd_nodes_pds: a generation outgrew the scratch buffers");
    return RBFFD_ERR_CUDA;
}
