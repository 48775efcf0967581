// rbffd_knn: support selection (Sec. II, text after Eq. 1) - for each centre
// the n nearest nodes, centre included, ordered by the key (d2, node index).
//
// Two searches share the result's definition.  knn_fast (below) serves nearly
// every centre: it selects and orders candidates on FP32 distances with a
// proven error bound and forms FP64 distances only where that bound leaves
// the order open.  knn_kernel, all in FP64, serves the centres knn_fast hands
// back, grids too fine for FP32, and the allocation-free entry point.
//
// knn_kernel: nodes are binned into a uniform cell grid (about one node per
// cell; counting sort, ids ascending inside a cell).  One warp serves one
// centre.  It scans the cells of a box of Chebyshev radius r around the
// centre's cell, streaming candidates through a warp-local top-n (candidates
// that cannot beat the current n-th key are dropped by a ballot; survivors are
// merged by exact rank), then grows the box until every node outside it is
// provably farther than the current n-th key.  Growing only scans the new
// shell.  Squared distances are formed exactly like the definition
// (fl(fl(dx*dx) + fl(dy*dy) ...), no contraction), so ties resolve by index
// and the result is bit-identical to any exact implementation.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace rbffd {

static constexpr int KNN_NMAX = 128;
static constexpr int KNN_BUF = 64;
static constexpr int KNN_WARPS = 4;

// distances are kept as the IEEE bits of d2: for non-negative doubles the
// unsigned integer order is the numeric order, so the (d2, index) key
// comparisons of the merges run on the integer pipes, not the FP64 pipe
struct KnnSmem {
    unsigned long long bd[2][KNN_NMAX];
    int32_t bj[2][KNN_NMAX];
    unsigned long long cd[KNN_BUF];
    int32_t cj[KNN_BUF];
    int32_t rb[32], rpre[32];   // range begin, inclusive prefix of lengths
};

struct KnnArgs {
    const double* xyz;
    int64_t N;
    int d;
    const int32_t* centres;
    int64_t nc;
    int n;
    int32_t* idx;
    GridGeom g;
    const int32_t* cell_start;
    const int32_t* sorted;
    const uint8_t* cand;   // NULL, or only nodes with cand != 0 (and the centre) qualify
    int r0;
    int* err;
    const int32_t* which;  // NULL, or the positions in `centres` to serve (nc of them)
    double margin;         // cells by which a node may lie outside its cell's bounds
};

__device__ __forceinline__ bool kless(unsigned long long da, int32_t ja, unsigned long long db,
                                      int32_t jb) {
    return da < db || (da == db && ja < jb);
}

__device__ __forceinline__ double sqdist(const double* xyz, int64_t N, int d, int32_t j,
                                         const double* q) {
    double s = 0.0;
    for (int a = 0; a < d; ++a) {
        double t = __dsub_rn(xyz[(int64_t)a * N + j], q[a]);
        double sq = __dmul_rn(t, t);
        s = (a == 0) ? sq : __dadd_rn(s, sq);
    }
    return s;
}

// merge best[cur] (nb entries) with the buffer (nbuf) into best[cur^1]; keep n
__device__ void knn_merge(KnnSmem& sm, int& cur, int& nb, int nbuf, int n, int lane) {
    __syncwarp();
    int L = nb + nbuf;
    for (int e = lane; e < L; e += 32) {
        unsigned long long de = e < nb ? sm.bd[cur][e] : sm.cd[e - nb];
        int32_t je = e < nb ? sm.bj[cur][e] : sm.cj[e - nb];
        int rank = 0;
        for (int f = 0; f < nb; ++f) rank += kless(sm.bd[cur][f], sm.bj[cur][f], de, je);
        for (int f = 0; f < nbuf; ++f) rank += kless(sm.cd[f], sm.cj[f], de, je);
        if (rank < n) {
            sm.bd[cur ^ 1][rank] = de;
            sm.bj[cur ^ 1][rank] = je;
        }
    }
    __syncwarp();
    cur ^= 1;
    nb = L < n ? L : n;
}

__global__ void __launch_bounds__(32 * KNN_WARPS) knn_kernel(KnnArgs A) {
    __shared__ KnnSmem smem[KNN_WARPS];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    KnnSmem& sm = smem[wib];
    const GridGeom& g = A.g;
    const int d = A.d, n = A.n;
    const int last = d - 1;   // contiguous axis of the row-major cell grid
    const int64_t warps = (int64_t)gridDim.x * KNN_WARPS;

    for (int64_t wi = (int64_t)blockIdx.x * KNN_WARPS + wib; wi < A.nc; wi += warps) {
        const int64_t qi = A.which ? A.which[wi] : wi;
        const int32_t c = A.centres[qi];
        double q[3] = {0, 0, 0};
        int cc[3] = {0, 0, 0};
        for (int a = 0; a < d; ++a) {
            q[a] = A.xyz[(int64_t)a * A.N + c];
            cc[a] = cell_coord(q[a], g.org[a], g.cs, g.G[a]);
        }
        int cur = 0, nb = 0, nbuf = 0;
        int r = A.r0, prev = -1;
        bool done = false;
        for (int guard = 0; guard < 1 << 20 && !done; ++guard) {
            // rows of the box: all axes but the last; each row gives two slots
            // (left and right of the previous box, or the whole row)
            int side = 2 * r + 1;
            int64_t nrows = 1;
            for (int a = 0; a < last; ++a) nrows *= side;
            int64_t nslots = 2 * nrows;
            for (int64_t s0 = 0; s0 < nslots; s0 += 32) {
                // lane k describes slot s0 + k as a range of `sorted`
                int64_t s = s0 + lane;
                int32_t beg = 0, len = 0;
                if (s < nslots) {
                    int64_t row = s >> 1;
                    int half = (int)(s & 1);
                    bool ok = true, inside_prev = (prev >= 0);
                    int64_t cell_row = 0;
                    int64_t rem = row;
                    int crow[3] = {0, 0, 0};
                    for (int a = last - 1; a >= 0; --a) {
                        crow[a] = cc[a] - r + (int)(rem % side);
                        rem /= side;
                    }
                    for (int a = 0; a < last; ++a) {
                        if (crow[a] < 0 || crow[a] >= g.G[a]) ok = false;
                        int dd = crow[a] - cc[a];
                        if (dd < -prev || dd > prev) inside_prev = false;
                        cell_row = cell_row * g.G[a] + crow[a];
                    }
                    int lo = cc[last] - r, hi = cc[last] + r;
                    if (inside_prev) {
                        if (half == 0) hi = cc[last] - prev - 1;
                        else lo = cc[last] + prev + 1;
                    } else if (half == 1) {
                        ok = false;
                    }
                    if (lo < 0) lo = 0;
                    if (hi > g.G[last] - 1) hi = g.G[last] - 1;
                    if (ok && lo <= hi) {
                        int64_t base = cell_row * g.G[last];
                        beg = A.cell_start[base + lo];
                        len = A.cell_start[base + hi + 1] - beg;
                    }
                }
                int32_t pre = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int32_t t = __shfl_up_sync(0xffffffffu, pre, o);
                    if (lane >= o) pre += t;
                }
                sm.rb[lane] = beg;
                sm.rpre[lane] = pre;
                int32_t total = __shfl_sync(0xffffffffu, pre, 31);
                __syncwarp();
                for (int32_t v0 = 0; v0 < total; v0 += 32) {
                    if (nbuf + 32 > KNN_BUF) {
                        knn_merge(sm, cur, nb, nbuf, n, lane);
                        nbuf = 0;
                    }
                    int32_t v = v0 + lane;
                    bool acc = false;
                    unsigned long long dv = 0;
                    int32_t jv = 0;
                    if (v < total) {
                        int k = 0;   // first slot with inclusive prefix > v
                        for (int step = 16; step > 0; step >>= 1)
                            if (sm.rpre[k + step - 1] <= v) k += step;
                        int32_t off = v - (k ? sm.rpre[k - 1] : 0);
                        jv = A.sorted[sm.rb[k] + off];
                        dv = (unsigned long long)__double_as_longlong(sqdist(A.xyz, A.N, d, jv, q));
                        acc = (nb < n) || kless(dv, jv, sm.bd[cur][n - 1], sm.bj[cur][n - 1]);
                        if (A.cand && !A.cand[jv] && jv != c) acc = false;
                    }
                    unsigned m = __ballot_sync(0xffffffffu, acc);
                    if (acc) {
                        int p = nbuf + __popc(m & ((1u << lane) - 1u));
                        sm.cd[p] = dv;
                        sm.cj[p] = jv;
                    }
                    nbuf += __popc(m);
                }
                __syncwarp();
            }
            if (nbuf > 0) {
                knn_merge(sm, cur, nb, nbuf, n, lane);
                nbuf = 0;
            }
            // termination: every node outside the box is farther than the n-th key
            double bound = INFINITY;
            bool whole = true;
            for (int a = 0; a < d; ++a) {
                int lo = cc[a] - r, hi = cc[a] + r;
                if (lo > 0) {
                    whole = false;
                    bound = fmin(bound, q[a] - (g.org[a] + (double)lo * g.cs));
                }
                if (hi < g.G[a] - 1) {
                    whole = false;
                    bound = fmin(bound, (g.org[a] + (double)(hi + 1) * g.cs) - q[a]);
                }
            }
            if (whole) {
                done = true;
            } else if (nb == n) {
                double be = bound - A.margin * g.cs;
                double worst = __longlong_as_double((long long)sm.bd[cur][n - 1]);
                if (be > 0.0 && worst < be * be * (1.0 - 1e-12)) {
                    done = true;
                } else {
                    int need = (int)ceil(sqrt(worst) / g.cs) + 1;
                    prev = r;
                    r = need > r + 1 ? need : r + 1;
                }
            } else {
                prev = r;
                r = r + 1;
            }
        }
        if (!done && lane == 0) atomicExch(A.err, 1);
        if (done && nb < n && lane == 0) atomicExch(A.err, 2);   // too few candidates
        __syncwarp();
        for (int k = lane; k < n; k += 32)
            A.idx[qi * n + k] = k < nb ? sm.bj[cur][k] : -1;
        __syncwarp();
    }
}


// ---------------------------------------------------------------------------
// knn_fast: the same supports from FP32 distances wherever those decide.
//
// Coordinates in cell units, x' = fl32((x - org) / cs), carry an absolute
// error of at most delta = 2^(k-25) for grids of up to 2^k cells an axis, so
// an FP32 squared distance differs from the true one (in cells) by at most
// eps (knn_eps).  One warp serves one centre:
//  1. every node of the cells that meet the ball of radius R around the
//     centre (R from the mean density of one node per cell) is a candidate;
//     those with d2 < R^2 are kept, and counted in 256 equal bins of d2;
//  2. the first bin b at which the count reaches n bounds the support: no
//     node of the support lies above bin b + 1 (bins are wider than 4 eps).
//     Where b > 254 or fewer than n candidates came, R grows and the scan
//     starts again;
//  3. the candidates up to bin b + 1 are placed by bin (a counting sort), and
//     each one's rank is the number of entries in the bins below its
//     neighbours' plus the smaller ones among its own and the two adjacent
//     bins.  Two entries whose FP32 values differ by more than 2 eps are in
//     that order; the rest - about 0.5 % on jittered nodes, all of them on
//     exact grids - are ordered by their FP64 (d2, index) keys, formed as the
//     definition says.
// What bounds it: instruction issue (the FP64 pipe, which the all-FP64 search
// kept busy with every candidate's distance, takes one candidate in 200).
// Centres whose candidates or support candidates overflow the warp's arrays,
// or whose ball outgrows the node set, go to a list that knn_kernel serves.
// Whole call, knn_kernel alone -> knn_fast: jittered squares of 1M nodes 3.60
// -> 1.04 ms (n = 12), 4.35 -> 1.26 (30), 7.84 -> 1.61 (56); cube of 1M nodes
// 6.95 -> 1.27 (20), 24.8 -> 2.30 (70); 1M random points 4.41 -> 1.36 (30); an
// exact grid of 1M, every distance tied, 4.35 -> 2.23 (30); 10k nodes 0.18 ->
// 0.12 (12).  knn_kernel spent its time ranking every buffered candidate
// against every other (64-bit keys) and on FP64 distances and divisions.
// ---------------------------------------------------------------------------
static constexpr int KF_WARPS = 4;
static constexpr int KF_CAND = 384;   // candidates of one centre
static constexpr int KF_SEL = 192;    // candidates placed for ranking
static constexpr int KF_BINS = 256;

struct KnnFast {
    const double* xyz;
    int64_t N;
    const int32_t* centres;
    int64_t nc;
    int n;
    int32_t* idx;
    const float4* node;        // [N] cell-unit coordinates by node id
    const float4* sorted;      // [N] the same by cell, w = node id (as bits)
    const int32_t* cell_start;
    const uint8_t* cand;
    int G[3];
    float R0, Rmax;            // first radius, radius that holds the whole set (cells)
    float eps_r, eps_0;        // eps(R) = eps_r R^2 + eps_0 R + eps_0^2
    int32_t* left;             // centres handed back, *nleft of them
    int* nleft;
};

struct KnnFastSmem {
    int32_t hist[KF_BINS];
    unsigned long long key[KF_SEL];
    int32_t id[KF_SEL];
    float a[KF_SEL];
    uint8_t bin[KF_SEL];
    float ca[KF_CAND];
    int32_t cp[KF_CAND];
    int32_t rb[32], rpre[32];
};

// cell coordinate of a cell-unit coordinate: one map for binning and search
__device__ __forceinline__ int fast_cell(float x, int G) {
    const int c = (int)x;   // x >= 0
    return c < G ? c : G - 1;
}

// cell-unit coordinates, the cell's count and the node's place in its cell
__global__ void fast_cells(const double* __restrict__ xyz, int64_t N, int d, double3 org,
                           double inv, int3 G, float4* __restrict__ node,
                           int32_t* __restrict__ key, int32_t* __restrict__ place,
                           int32_t* __restrict__ count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        float x[3] = {0.f, 0.f, 0.f};
        x[0] = fmaxf(0.f, (float)__dmul_rn(__dsub_rn(xyz[i], org.x), inv));
        if (d > 1) x[1] = fmaxf(0.f, (float)__dmul_rn(__dsub_rn(xyz[N + i], org.y), inv));
        if (d > 2) x[2] = fmaxf(0.f, (float)__dmul_rn(__dsub_rn(xyz[2 * N + i], org.z), inv));
        int c = fast_cell(x[0], G.x);
        if (d > 1) c = c * G.y + fast_cell(x[1], G.y);
        if (d > 2) c = c * G.z + fast_cell(x[2], G.z);
        node[i] = make_float4(x[0], x[1], x[2], __int_as_float((int)i));
        key[i] = c;
        place[i] = atomicAdd(&count[c], 1);
    }
}

// nodes into cell order (any order inside a cell: the search ranks exactly)
__global__ void fast_scatter(const float4* __restrict__ node, int64_t N,
                             const int32_t* __restrict__ key, const int32_t* __restrict__ place,
                             const int32_t* __restrict__ start, float4* __restrict__ sorted,
                             int32_t* __restrict__ ids) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int p = start[key[i]] + place[i];
        sorted[p] = node[i];
        ids[p] = (int32_t)i;
    }
}

template <int D>
__global__ void __launch_bounds__(32 * KF_WARPS) knn_fast(KnnFast A) {
    extern __shared__ __align__(16) unsigned char kf_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    KnnFastSmem& sm = reinterpret_cast<KnnFastSmem*>(kf_smem)[wib];
    const unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const int n = A.n;
    const int64_t warps = (int64_t)gridDim.x * KF_WARPS;
    for (int64_t qi = (int64_t)blockIdx.x * KF_WARPS + wib; qi < A.nc; qi += warps) {
        const int32_t c = A.centres[qi];
        const float4 qf = A.node[c];
        const float q[3] = {qf.x, qf.y, qf.z};
        float R = A.R0;
        bool served = false;
        for (int tries = 0; tries < 24; ++tries) {
            const float R2 = R * R, scale = (float)KF_BINS / R2;
            // the margin covers the rounding of q +- R and of the nodes' cells
            const float Rm = R + 4e-3f + 1e-6f * R;
            {
                int4* h4 = reinterpret_cast<int4*>(sm.hist);
                h4[lane] = make_int4(0, 0, 0, 0);
                h4[lane + 32] = make_int4(0, 0, 0, 0);
            }
            __syncwarp();
            // rows of cells along the last axis that meet the ball
            int lo[2] = {0, 0}, cnt[2] = {1, 1};
#pragma unroll
            for (int a = 0; a + 1 < D; ++a) {
                lo[a] = max(0, (int)floorf(q[a] - Rm));
                cnt[a] = min(A.G[a] - 1, (int)floorf(q[a] + Rm)) - lo[a] + 1;
            }
            const int nrows = cnt[0] * cnt[1];
            int ncand = 0;
            for (int s0 = 0; s0 < nrows && ncand <= KF_CAND; s0 += 32) {
                const int row = s0 + lane;
                int32_t beg = 0, len = 0;
                if (row < nrows) {
                    int cr[2] = {row, 0};
                    if (D == 3) {
                        cr[0] = row / cnt[1];
                        cr[1] = row - cr[0] * cnt[1];
                    }
                    float away = 0.f;
                    int64_t base = 0;
#pragma unroll
                    for (int a = 0; a + 1 < D; ++a) {
                        const int ca = lo[a] + cr[a];
                        const float gap = fmaxf(0.f, fmaxf((float)ca - q[a], q[a] - (float)(ca + 1)));
                        away += gap * gap;
                        base = base * A.G[a] + ca;
                    }
                    base *= A.G[D - 1];
                    const float rest = Rm * Rm - away;
                    if (rest >= 0.f) {
                        const float w = sqrtf(rest) + 4e-3f;
                        const int l = max(0, (int)floorf(q[D - 1] - w));
                        const int h = min(A.G[D - 1] - 1, (int)floorf(q[D - 1] + w));
                        if (l <= h) {
                            beg = __ldg(A.cell_start + base + l);
                            len = __ldg(A.cell_start + base + h + 1) - beg;
                        }
                    }
                }
                int32_t pre = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t t = __shfl_up_sync(FULL, pre, o);
                    if (lane >= o) pre += t;
                }
                sm.rb[lane] = beg - (pre - len);   // position = rb + running number
                sm.rpre[lane] = pre;
                const int32_t total = __shfl_sync(FULL, pre, 31);
                __syncwarp();
                for (int32_t v0 = 0; v0 < total; v0 += 32) {
                    const int32_t v = v0 + lane;
                    bool in = false;
                    float d2 = 0.f;
                    int32_t p = 0;
                    if (v < total) {
                        int k = 0;   // first row with inclusive prefix > v
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            if (sm.rpre[k + step - 1] <= v) k += step;
                        p = sm.rb[k] + v;
                        const float4 x = __ldg(A.sorted + p);
                        const float dx = x.x - q[0];
                        d2 = dx * dx;
                        if (D > 1) {
                            const float dy = x.y - q[1];
                            d2 += dy * dy;
                        }
                        if (D > 2) {
                            const float dz = x.z - q[2];
                            d2 += dz * dz;
                        }
                        in = d2 < R2;
                        if (in && A.cand) {
                            const int32_t j = __float_as_int(x.w);
                            in = A.cand[j] || j == c;
                        }
                    }
                    const unsigned m = __ballot_sync(FULL, in);
                    if (in) {
                        const int at = ncand + __popc(m & below);
                        if (at < KF_CAND) {
                            sm.ca[at] = d2;
                            sm.cp[at] = p;
                            atomicAdd(&sm.hist[min(KF_BINS - 1, (int)(d2 * scale))], 1);
                        }
                    }
                    ncand += __popc(m);
                    if (ncand > KF_CAND) break;
                }
                __syncwarp();
            }
            if (ncand > KF_CAND) break;   // too dense for the arrays
            if (ncand < n) {
                if (R > A.Rmax) break;    // fewer than n candidates in all
                float f = D == 1 ? (float)n / (float)max(ncand, 1)
                          : D == 2 ? sqrtf((float)n / (float)max(ncand, 1))
                                   : cbrtf((float)n / (float)max(ncand, 1));
                R *= fminf(fmaxf(f * 1.06f, 1.1f), 2.f);
                continue;
            }
            // bins -> exclusive starts; the first bin whose inclusive count reaches n
            int4* h4 = reinterpret_cast<int4*>(sm.hist);
            int4 ha = h4[2 * lane], hb = h4[2 * lane + 1];
            const int sum = ha.x + ha.y + ha.z + ha.w + hb.x + hb.y + hb.z + hb.w;
            int inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += t;
            }
            int st[9];
            st[0] = inc - sum;
            st[1] = st[0] + ha.x;
            st[2] = st[1] + ha.y;
            st[3] = st[2] + ha.z;
            st[4] = st[3] + ha.w;
            st[5] = st[4] + hb.x;
            st[6] = st[5] + hb.y;
            st[7] = st[6] + hb.z;
            st[8] = st[7] + hb.w;
            h4[2 * lane] = make_int4(st[0], st[1], st[2], st[3]);
            h4[2 * lane + 1] = make_int4(st[4], st[5], st[6], st[7]);
            int fb = 0;   // bins of this lane whose inclusive count is below n
#pragma unroll
            for (int k = 1; k <= 8; ++k) fb += st[k] < n;
            const unsigned reach = __ballot_sync(FULL, fb < 8);
            const int src = __ffs(reach) - 1;
            const int b = 8 * src + __shfl_sync(FULL, fb, src);
            __syncwarp();
            if (b > KF_BINS - 2) {
                R *= 1.05f;
                continue;
            }
            const int last = b + 1;
            const int S = last + 1 < KF_BINS ? sm.hist[last + 1] : ncand;
            if (S > KF_SEL) break;
            __syncwarp();
            // place: afterwards hist[k] is the end of bin k for k <= last
            for (int i = lane; i < ncand; i += 32) {
                const float d2 = sm.ca[i];
                const int bi = min(KF_BINS - 1, (int)(d2 * scale));
                if (bi <= last) {
                    const int at = atomicAdd(&sm.hist[bi], 1);
                    sm.a[at] = d2;
                    sm.id[at] = __float_as_int(__ldg(&A.sorted[sm.cp[i]].w));
                    sm.bin[at] = (uint8_t)bi;
                }
            }
            __syncwarp();
            const float two_eps = 2.f * (A.eps_r * R2 + A.eps_0 * R + A.eps_0 * A.eps_0);
            int32_t* out = sm.cp;   // the candidates' positions are no longer needed
            bool any_open = false;
            for (int p0 = 0; p0 < S; p0 += 32) {
                const int p = p0 + lane;
                int rank = n;
                bool open = false;
                if (p < S) {
                    const int bi = sm.bin[p];
                    const float ap = sm.a[p];
                    const int w0 = bi >= 2 ? sm.hist[bi - 2] : 0;
                    const int w1 = sm.hist[min(bi + 1, last)];
                    rank = w0;
                    for (int e = w0; e < w1; ++e) {
                        const float t = sm.a[e] - ap;
                        if (fabsf(t) <= two_eps) open = open || e != p;
                        else rank += t < 0.f;
                    }
                    if (!open && rank < n) out[rank] = sm.id[p];
                }
                // an open pair is open from both sides, so both keys get formed
                if (__any_sync(FULL, open)) {
                    any_open = true;
                    if (open) {
                        double qx[3];
#pragma unroll
                        for (int a = 0; a < D; ++a) qx[a] = __ldg(A.xyz + (int64_t)a * A.N + c);
                        sm.key[p] = (unsigned long long)__double_as_longlong(
                            sqdist(A.xyz, A.N, D, sm.id[p], qx));
                    }
                }
            }
            __syncwarp();
            for (int p = lane; any_open && p < S; p += 32) {
                const int bi = sm.bin[p];
                const float ap = sm.a[p];
                const int w0 = bi >= 2 ? sm.hist[bi - 2] : 0;
                const int w1 = sm.hist[min(bi + 1, last)];
                int rank = w0;
                bool open = false;
                for (int e = w0; e < w1; ++e) {
                    const float t = sm.a[e] - ap;
                    if (fabsf(t) > two_eps) {
                        rank += t < 0.f;
                    } else if (e != p) {
                        open = true;
                        rank += kless(sm.key[e], sm.id[e], sm.key[p], sm.id[p]);
                    }
                }
                if (open && rank < n) out[rank] = sm.id[p];
            }
            __syncwarp();
            for (int k = lane; k < n; k += 32) A.idx[qi * n + k] = out[k];
            __syncwarp();
            served = true;
            break;
        }
        if (!served && lane == 0) A.left[atomicAdd(A.nleft, 1)] = (int32_t)qi;
        __syncwarp();
    }
}

}  // namespace rbffd

using namespace rbffd;

// 8-byte-aligned carving of one allocation
struct Carve {
    size_t used = 0;
    size_t take(size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) / 256 * 256;
        return at;
    }
};

static int knn_impl(const double* xyz, int64_t N, int d, const uint8_t* cand,
                    const int32_t* centres, int64_t nc, int n, int32_t* idx, void* stream) {
    RBFFD_ARG(nc >= 0, "rbffd_knn: negative centre count");
    if (nc == 0) return RBFFD_OK;
    RBFFD_ARG(xyz && centres && idx, "rbffd_knn: NULL argument");
    RBFFD_ARG(d >= 1 && d <= 3, "rbffd_knn: d must be 1, 2 or 3");
    RBFFD_ARG(N >= 1 && N < (int64_t(1) << 31), "rbffd_knn: bad N");
    RBFFD_ARG(n >= 1 && n <= KNN_NMAX && n <= N, "rbffd_knn: need 1 <= n <= min(N, %d)",
              KNN_NMAX);
    cudaStream_t s = as_stream(stream);
    double lo[3], hi[3];
    int st = bounding_box(xyz, N, d, lo, hi, s);
    if (st) return st;
    GridGeom g = make_grid(d, lo, hi, N, 1.0);
    const int64_t ncell = g.ncell();
    // initial search radius in cells: a ball of n nodes at mean density (knn_fast
    // adds a margin for its spread; 0.0-0.5 / sqrt n and 0.1-0.2 cells measured
    // within 4 % of each other on jittered and on random sets)
    const double per_cell = (double)N / (double)ncell;
    const double ball[4] = {0, 2.0, M_PI, 4.0 * M_PI / 3.0};
    const double rad = pow((double)n / (ball[d] * per_cell), 1.0 / d);
    // knn_fast where its FP32 error bound is a quarter of its bins' width or
    // less (grids of up to 2^13 or 2^14 cells an axis); beyond that the bins no
    // longer bound a node's rank, whatever the speed
    const int Gmax = std::max(g.G[0], std::max(g.G[1], g.G[2]));
    int k = 0;
    while ((int64_t(1) << k) < Gmax) ++k;
    const double delta = ldexp(1.0, k - 25), rd = sqrt((double)d);
    KnnFast F;
    F.eps_r = (float)(1.25 * (2.0 * rd + 2.0) * ldexp(1.0, -23));
    F.eps_0 = (float)(1.25 * 4.0 * rd * delta);
    F.R0 = (float)(rad * (1.0 + 0.2 / sqrt((double)n)) + 0.1);
    F.Rmax = 2.f;
    for (int a = 0; a < d; ++a) F.Rmax += (float)g.G[a];
    const double eps =
        F.eps_r * (double)F.R0 * F.R0 + (double)F.eps_0 * F.R0 + (double)F.eps_0 * F.eps_0;
    bool fast = 4.0 * eps < (double)F.R0 * F.R0 / KF_BINS;

    Carve cv;
    const size_t o_start = cv.take(sizeof(int32_t) * (size_t)(ncell + 1));
    const size_t o_ids = cv.take(sizeof(int32_t) * (size_t)N);
    const size_t o_flags = cv.take(2 * sizeof(int));   // err, centres left to knn_kernel
    const size_t slow_bytes = cv.used;
    const size_t o_count = fast ? cv.take(sizeof(int32_t) * (size_t)(ncell + 1)) : 0;
    const size_t o_tmp = fast ? cv.take(sizeof(int64_t) * (size_t)scan_tmp_elems(ncell)) : 0;
    const size_t o_key = fast ? cv.take(sizeof(int32_t) * (size_t)N) : 0;
    const size_t o_place = fast ? cv.take(sizeof(int32_t) * (size_t)N) : 0;
    const size_t o_node = fast ? cv.take(sizeof(float4) * (size_t)N) : 0;
    const size_t o_sorted = fast ? cv.take(sizeof(float4) * (size_t)N) : 0;
    const size_t o_left = fast ? cv.take(sizeof(int32_t) * (size_t)nc) : 0;
    Scratch mem;
    cudaError_t e = mem.alloc(cv.used, s);
    if (e == cudaErrorMemoryAllocation && fast) {   // knn_kernel needs a seventh of it
        cudaGetLastError();
        fast = false;
        e = mem.alloc(slow_bytes, s);
    }
    RBFFD_CHECK_CUDA(e);
    char* base = mem.as<char>();
    int32_t* start = reinterpret_cast<int32_t*>(base + o_start);
    int32_t* ids = reinterpret_cast<int32_t*>(base + o_ids);
    int* flags = reinterpret_cast<int*>(base + o_flags);
    RBFFD_CHECK_CUDA(cudaMemsetAsync(flags, 0, 2 * sizeof(int), s));
    const int sms = device_sm_count();
    int hf[2] = {0, 0};
    KnnArgs A;
    A.which = nullptr;
    A.margin = 1e-6;
    int64_t rest = nc;   // centres for knn_kernel
    if (fast) {
        int32_t* count = reinterpret_cast<int32_t*>(base + o_count);
        int32_t* key = reinterpret_cast<int32_t*>(base + o_key);
        int32_t* place = reinterpret_cast<int32_t*>(base + o_place);
        float4* node = reinterpret_cast<float4*>(base + o_node);
        float4* sorted = reinterpret_cast<float4*>(base + o_sorted);
        RBFFD_CHECK_CUDA(cudaMemsetAsync(count, 0, sizeof(int32_t) * (size_t)(ncell + 1), s));
        fast_cells<<<sms * 8, 256, 0, s>>>(xyz, N, d, make_double3(g.org[0], g.org[1], g.org[2]),
                                           1.0 / g.cs, make_int3(g.G[0], g.G[1], g.G[2]), node,
                                           key, place, count);
        RBFFD_CHECK_CUDA(cudaGetLastError());
        RBFFD_CHECK_CUDA(exclusive_scan_i32(count, start, ncell,
                                            reinterpret_cast<int64_t*>(base + o_tmp), s));
        fast_scatter<<<sms * 8, 256, 0, s>>>(node, N, key, place, start, sorted, ids);
        F.xyz = xyz;
        F.N = N;
        F.centres = centres;
        F.nc = nc;
        F.n = n;
        F.idx = idx;
        F.node = node;
        F.sorted = sorted;
        F.cell_start = start;
        F.cand = cand;
        for (int a = 0; a < 3; ++a) F.G[a] = g.G[a];
        F.left = reinterpret_cast<int32_t*>(base + o_left);
        F.nleft = flags + 1;
        void (*fn)(KnnFast) = d == 1 ? knn_fast<1> : d == 2 ? knn_fast<2> : knn_fast<3>;
        const int smem = KF_WARPS * (int)sizeof(KnnFastSmem);
        const int64_t blocks = (nc + KF_WARPS - 1) / KF_WARPS;
        fn<<<(unsigned)std::min<int64_t>(blocks, (int64_t)sms * 64), 32 * KF_WARPS, smem, s>>>(F);
        RBFFD_CHECK_CUDA(cudaGetLastError());
        RBFFD_CHECK_CUDA(cudaMemcpyAsync(hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, s));
        RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
        rest = hf[1];
        A.which = F.left;
        // nodes were put into cells by their FP32 coordinates (error below
        // 2^-11 cells, see `fast`)
        A.margin = 0.01;
    } else {
        st = build_cell_lists(xyz, N, g, start, ids, s);
        if (st) return st;
    }
    if (rest > 0) {
        A.xyz = xyz;
        A.N = N;
        A.d = d;
        A.centres = centres;
        A.nc = rest;
        A.n = n;
        A.idx = idx;
        A.g = g;
        A.cell_start = start;
        A.sorted = ids;
        A.cand = cand;
        A.r0 = (int)ceil(rad) > 1 ? (int)ceil(rad) : 1;
        A.err = flags;
        const int64_t blocks = (rest + KNN_WARPS - 1) / KNN_WARPS;
        const int64_t cap = (int64_t)sms * 64;
        knn_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 32 * KNN_WARPS, 0, s>>>(A);
        RBFFD_CHECK_CUDA(cudaGetLastError());
        RBFFD_CHECK_CUDA(cudaMemcpyAsync(hf, flags, sizeof(int), cudaMemcpyDeviceToHost, s));
        RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
    }
    if (hf[0] == 2) {
        set_error("rbffd_knn: fewer than n candidate nodes");
        return RBFFD_ERR_ARG;
    }
    if (hf[0]) {
        set_error("rbffd_knn: ring search did not terminate");
        return RBFFD_ERR_CAPACITY;
    }
    return RBFFD_OK;
}

extern "C" int rbffd_knn(const double* xyz, int64_t N, int d, const int32_t* centres, int64_t nc,
                         int n, int32_t* idx, void* stream) {
    clear_error();
    return knn_impl(xyz, N, d, nullptr, centres, nc, n, idx, stream);
}

extern "C" int rbffd_knn_masked(const double* xyz, int64_t N, int d, const uint8_t* cand,
                                const int32_t* centres, int64_t nc, int n, int32_t* idx,
                                void* stream) {
    clear_error();
    RBFFD_ARG(cand != nullptr || nc == 0, "rbffd_knn_masked: NULL candidate mask");
    return knn_impl(xyz, N, d, cand, centres, nc, n, idx, stream);
}



// ---------------------------------------------------------------------------
// rbffd_knn_noalloc: the same support selection for callers that cannot
// allocate device memory while they run.  Its working memory is one
// file-scope __device__ array of fixed size (every GPU that loads the library
// holds it until the process exits), reached from host code through the
// address that cudaGetSymbolAddress returns for the current device.
// ---------------------------------------------------------------------------
namespace rbffd {

static constexpr int64_t NA_MAX_NODES = RBFFD_KNN_NOALLOC_MAX_NODES;
static constexpr int64_t NA_MAX_CELLS = 2 * NA_MAX_NODES;
static constexpr size_t na_round(size_t b) { return (b + 255) / 256 * 256; }
static constexpr int NA_BBOX_BLOCKS = 256;
// byte offsets of the regions inside the scratch array (each 256-aligned)
static constexpr size_t NA_OFF_PART = 0;                                       // bbox partials
static constexpr size_t NA_OFF_ERR = NA_OFF_PART + na_round(sizeof(double) * 6 * NA_BBOX_BLOCKS);
static constexpr size_t NA_OFF_START = NA_OFF_ERR + 256;                         // cell starts
static constexpr size_t NA_OFF_COUNT = NA_OFF_START + na_round(4 * (NA_MAX_CELLS + 1));
static constexpr size_t NA_OFF_TMP = NA_OFF_COUNT + na_round(4 * (NA_MAX_CELLS + 1));
static constexpr int64_t NA_TMP_ELEMS = (NA_MAX_CELLS + 2047) / 2048 + 1;      // scan tiles
static constexpr size_t NA_OFF_KEY = NA_OFF_TMP + na_round(8 * NA_TMP_ELEMS);
static constexpr size_t NA_OFF_SORTED = NA_OFF_KEY + na_round(4 * NA_MAX_NODES);
static constexpr size_t NA_BYTES = NA_OFF_SORTED + na_round(4 * NA_MAX_NODES);

static __device__ __align__(256) unsigned char g_knn_noalloc_scratch[NA_BYTES];

// device address of the scratch array for the current device, looked up once
// per device (host code may not use the array's name as a device pointer)
static int noalloc_scratch(unsigned char** out) {
    static std::mutex mu;
    static void* addr[128] = {};
    int dev = 0;
    RBFFD_CHECK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 128) {
        set_error("rbffd_knn_noalloc: device ordinal %d out of range", dev);
        return RBFFD_ERR_ARG;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_knn_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            set_error("rbffd_knn_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            return RBFFD_ERR_CUDA;
        }
        addr[dev] = p;
    }
    *out = static_cast<unsigned char*>(addr[dev]);
    return RBFFD_OK;
}

}  // namespace rbffd

extern "C" int rbffd_knn_noalloc(const double* xyz, int64_t N, int d, const int32_t* centres,
                                 int64_t nc, int n, int32_t* idx, void* stream) {
    clear_error();
    RBFFD_ARG(nc >= 0, "rbffd_knn_noalloc: negative centre count");
    RBFFD_ARG(d >= 1 && d <= 3, "rbffd_knn_noalloc: d must be 1, 2 or 3");
    RBFFD_ARG(N >= 1, "rbffd_knn_noalloc: bad N");
    if (N > NA_MAX_NODES) {
        set_error("rbffd_knn_noalloc: %lld nodes exceed the fixed scratch limit of %lld "
                  "(use rbffd_knn)", (long long)N, (long long)NA_MAX_NODES);
        return RBFFD_ERR_CAPACITY;
    }
    RBFFD_ARG(n >= 1 && n <= KNN_NMAX && n <= N, "rbffd_knn_noalloc: need 1 <= n <= min(N, %d)",
              KNN_NMAX);
    if (nc == 0) return RBFFD_OK;
    RBFFD_ARG(xyz && centres && idx, "rbffd_knn_noalloc: NULL argument");
    cudaStream_t s = as_stream(stream);
    unsigned char* base = nullptr;
    int st = noalloc_scratch(&base);
    if (st) return st;
    double* part = reinterpret_cast<double*>(base + NA_OFF_PART);
    int* err = reinterpret_cast<int*>(base + NA_OFF_ERR);
    int32_t* start = reinterpret_cast<int32_t*>(base + NA_OFF_START);
    int32_t* count = reinterpret_cast<int32_t*>(base + NA_OFF_COUNT);
    int64_t* tmp = reinterpret_cast<int64_t*>(base + NA_OFF_TMP);
    int32_t* key = reinterpret_cast<int32_t*>(base + NA_OFF_KEY);
    int32_t* sorted = reinterpret_cast<int32_t*>(base + NA_OFF_SORTED);

    // bounding box (partials in the scratch array, final reduction on the host)
    double hpart[NA_BBOX_BLOCKS * 6];
    bbox_partial<<<NA_BBOX_BLOCKS, 256, 0, s>>>(xyz, N, d, part);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    RBFFD_CHECK_CUDA(cudaMemcpyAsync(hpart, part, sizeof(hpart), cudaMemcpyDeviceToHost, s));
    RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
    double lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
        lo[a] = INFINITY;
        hi[a] = -INFINITY;
        for (int b = 0; b < NA_BBOX_BLOCKS; ++b) {
            lo[a] = fmin(lo[a], hpart[b * 6 + a]);
            hi[a] = fmax(hi[a], hpart[b * 6 + 3 + a]);
        }
        if (a >= d) lo[a] = hi[a] = 0.0;
    }
    for (int a = 0; a < d; ++a)
        RBFFD_ARG(isfinite(lo[a]) && isfinite(hi[a]), "rbffd_knn_noalloc: coordinates not finite");
    // cell grid of about one node per cell, coarsened to fit the fixed cell arrays
    GridGeom g = make_grid(d, lo, hi, N, 1.0);
    while (g.ncell() > NA_MAX_CELLS) {
        g.cs *= 1.25;
        for (int a = 0; a < d; ++a) g.G[a] = (int)floor((hi[a] - lo[a]) / g.cs) + 1;
    }
    const int64_t ncell = g.ncell();
    const int sms = device_sm_count();
    // the scratch keeps the previous call's contents: clear what must start at 0
    RBFFD_CHECK_CUDA(cudaMemsetAsync(count, 0, sizeof(int32_t) * (ncell + 1), s));
    RBFFD_CHECK_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    cells_key<<<sms * 8, 256, 0, s>>>(xyz, N, g, key);
    keys_count<<<sms * 8, 256, 0, s>>>(key, N, count);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    RBFFD_CHECK_CUDA(exclusive_scan_i32(count, start, ncell, tmp, s));
    RBFFD_CHECK_CUDA(cudaMemcpyAsync(count, start, sizeof(int32_t) * ncell,
                                     cudaMemcpyDeviceToDevice, s));
    cells_scatter<<<sms * 8, 256, 0, s>>>(N, key, count, sorted);
    cells_sort<<<sms * 8, 256, 0, s>>>(ncell, start, sorted);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    double per_cell = (double)N / (double)ncell;
    const double ball[4] = {0, 2.0, M_PI, 4.0 * M_PI / 3.0};
    double rad = pow((double)n / (ball[d] * per_cell), 1.0 / d);
    KnnArgs A;
    A.xyz = xyz;
    A.N = N;
    A.d = d;
    A.centres = centres;
    A.nc = nc;
    A.n = n;
    A.idx = idx;
    A.g = g;
    A.cell_start = start;
    A.sorted = sorted;
    A.cand = nullptr;
    A.which = nullptr;
    A.margin = 1e-6;
    A.r0 = (int)ceil(rad) > 1 ? (int)ceil(rad) : 1;
    A.err = err;
    int64_t blocks = (nc + KNN_WARPS - 1) / KNN_WARPS;
    int64_t cap = (int64_t)sms * 64;
    knn_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 32 * KNN_WARPS, 0, s>>>(A);
    RBFFD_CHECK_CUDA(cudaGetLastError());
    int herr = 0;
    RBFFD_CHECK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    RBFFD_CHECK_CUDA(cudaStreamSynchronize(s));
    if (herr) {
        set_error("rbffd_knn_noalloc: ring search did not terminate");
        return RBFFD_ERR_CAPACITY;
    }
    return RBFFD_OK;
}

