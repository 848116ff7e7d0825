// Pieces shared by the pair-symmetric evaluation kernels (pair_sym.cu, pair_fix.cu):
// the schedule of a launch, the ordered accumulation of the j-side sums (the
// protocol is described in pair_sym.cu) and the FP64 arithmetic of one block pair.
#pragma once

#include "common.cuh"
#include "pair_math.cuh"

namespace mh {

constexpr int kSymWarps = 4;
constexpr int kSymR = 32 * kSymWarps;     // bodies per block
constexpr int kFixRows = 3;               // rows per CTA of the fixed-point kernel
// Every form runs K rows of one chunk per CTA, one CTA per SM, and one
// accumulation chain (G = 1): fixed point K = 3, FP64 (P = 4, 5) K = 2, FP32-pair
// K = 6 where six rows' shared memory fits, else 4.  The turn computation takes
// any G (rows split into chains by row mod G); the plans use G = 1.

// Schedule of one launch (from SymPlan) and the ordered-accumulation words.
struct SymSched {
    int nB, D, C, Bc;      // C chunks: H consecutive ones share Bc distances
    int H;                 // chunk ch takes subtiles [ch % H, +1) kSymWarps / H of each of its blocks
    int G;                 // accumulation chains per j-slot: writer rows are split by row mod G
    int K;                 // rows per item (rows qK .. qK + K - 1 of one chunk)
    int cyclic;            // 1: one item per CTA, all resident; writers by descending distance
    int items;             // ceil(nB / K) * C
    unsigned *fetch;       // [1] next item to hand out (multi-wave order); reset by the launch's last fetch
    unsigned *count;       // [C][G][nB] writes done into j-slot (ch, g, J) in this launch; 0 between launches
    int *flag;             // status word: kFlagSymWait when a wait ran out
    unsigned long long wait_ns;   // limit of one wait
    unsigned bias;         // added to every awaited count (0 unless a host-injected fault asks otherwise)
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Thread 0: the CTA's next item (>= items once there is none).  The fetches of
// a launch number items + gridDim.x; the last one resets the counter.
__device__ __forceinline__ unsigned next_item(const SymSched &sc, int n)
{
    if (sc.cyclic) return n == 0 ? blockIdx.x : 0xffffffffu;
    const unsigned v = atomicAdd(sc.fetch, 1u);
    if (v == (unsigned)sc.items + gridDim.x - 1u) atomicExch(sc.fetch, 0u);
    return v;
}

// Distances [lo, hi) of the off-diagonal blocks of row chunk ch.
__host__ __device__ __forceinline__ void chunk_range(const SymSched &sc, int ch, int &lo, int &hi)
{
    const int b0 = ch / sc.H * sc.Bc;
    lo = b0 > 1 ? b0 : 1;
    hi = b0 + sc.Bc < sc.D + 1 ? b0 + sc.Bc : sc.D + 1;
}

// Whether row J - b (mod nB) adds into j-slot (ch, g, J) at distance b (a
// distance of chunk ch), i.e. evaluates that block and is in chain g; *before:
// whether it comes before row I (which evaluates J at distance bI) in the
// accumulation order.
__host__ __device__ __forceinline__ bool j_writer(const SymSched &sc, int J, int g, int b, int I, int bI,
                                                  bool *before)
{
    int r = J - b;
    if (r < 0) r += sc.nB;
    if ((sc.nB & 1) == 0 && b == sc.D && r >= sc.nB / 2) return false;   // rows >= nB/2 skip distance nB/2
    if (r % sc.G != g) return false;
    *before = sc.cyclic ? (b > bI) : (r < I);
    return true;
}

// The rows that add into j-slot (ch, g, J): I' = J - b (mod nB) for the
// distances b >= 1 of chunk ch that row I' evaluates, with I' = g (mod G).
// Returns how many there are and, in *rank, how many of them come before row I
// (which evaluates J at distance bI).  One thread.
__host__ __device__ __forceinline__ int j_writers(const SymSched &sc, int J, int ch, int g, int I, int bI,
                                                  int *rank)
{
    int lo, hi, nw = 0, rk = 0;
    chunk_range(sc, ch, lo, hi);
    for (int b = lo; b < hi; ++b) {
        bool before = false;
        if (j_writer(sc, J, g, b, I, bI, &before)) {
            ++nw;
            rk += before;
        }
    }
    *rank = rk;
    return nw;
}

// The same count by the 32 lanes of one warp (each lane takes every 32nd
// distance); every lane gets the result.
__device__ __forceinline__ int j_writers_warp(const SymSched &sc, int J, int ch, int g, int I, int bI, int *rank)
{
    int lo, hi, nw = 0, rk = 0;
    chunk_range(sc, ch, lo, hi);
    const int lane = threadIdx.x & 31;
    for (int b0 = lo; b0 < hi; b0 += 32) {
        bool before = false;
        const bool wr = b0 + lane < hi && j_writer(sc, J, g, b0 + lane, I, bI, &before);
        nw += __popc(__ballot_sync(0xffffffffu, wr));
        rk += __popc(__ballot_sync(0xffffffffu, wr && before));
    }
    *rank = rk;
    return nw;
}

// Thread 0: wait, bounded in time, until *c == want.
inline __device__ __noinline__ void wait_turn(const unsigned *c, unsigned want, const SymSched &sc)
{
    if (ld_acquire(c) == want) return;
    const unsigned long long t0 = now_ns();
    for (int it = 0;; ++it) {
        __nanosleep(it < 32 ? 20 : 200);
        if (ld_acquire(c) == want) return;
        if ((*(volatile int *)sc.flag & kFlagSymWait) || now_ns() - t0 > sc.wait_ns) {
            atomicOr(sc.flag, kFlagSymWait);
            return;
        }
    }
}

// Shared-memory words of one CTA for the ordered flush.
struct FlushSmem {
    int item, rank, next, ready;
    unsigned zero;        // bit g: j-slot (ch, g) of the item's own block has no writer
};

// Warp 0 at the start of item (I, ch): which of block I's j-slots of chunk ch
// no row adds into (they must hold zeros).
__device__ __forceinline__ unsigned unwritten_chains(const SymSched &sc, int I, int ch)
{
    unsigned z = 0;
    for (int g = 0; g < sc.G; ++g) {
        int rk;
        if (j_writers_warp(sc, I, ch, g, I, 0, &rk) == 0) z |= 1u << g;
    }
    return z;
}

// j-slot of chunk ch, chain g (the i-side slots come first).
__host__ __device__ __forceinline__ int64_t j_slot(const SymSched &sc, int ch, int g)
{
    return (int64_t)sc.C + (int64_t)ch * sc.G + g;
}

// Warp 0 of a row's threads (tu: thread index within the row) before row I's
// ordered flush into j-slot (ch, I mod G, J): publish the rank (0: this row
// writes first) and whether the turn has come (one look).
__device__ __forceinline__ void flush_rank(const SymSched &sc, FlushSmem &fs, int tu, int I, int J, int ch, int b)
{
    if (tu < 32) {
        const int g = I % sc.G;
        int rank = 0;
        const int nw = j_writers_warp(sc, J, ch, g, I, b, &rank);
        if (tu == 0) {
            fs.rank = rank;
            fs.next = rank + 1 == nw ? 0 : rank + 1;
            fs.ready = rank == 0 ||
                       ld_acquire(&sc.count[(j_slot(sc, ch, g) - sc.C) * sc.nB + J]) == (unsigned)rank + sc.bias;
        }
    }
}

// The row's thread 0: wait (bounded) for the turn flush_rank published, unless it had come.
__device__ __forceinline__ void flush_wait(const SymSched &sc, FlushSmem &fs, int tu, int I, int J, int ch)
{
    if (tu == 0 && !fs.ready) {
        wait_turn(&sc.count[(j_slot(sc, ch, I % sc.G) - sc.C) * sc.nB + J], (unsigned)fs.rank + sc.bias, sc);
        fs.ready = 1;
    }
}

// The row's thread 0 after the row's stores of the flush (behind the row's
// barrier): pass the turn on with a release store, which orders the row's
// stores before it (the last writer leaves the counter at 0).
__device__ __forceinline__ void flush_end(const SymSched &sc, const FlushSmem &fs, int tu, int I, int J, int ch)
{
    if (tu == 0)
        st_release(&sc.count[(j_slot(sc, ch, I % sc.G) - sc.C) * sc.nB + J], (unsigned)fs.next);
}

// Barrier of the n threads of row u of an item (barrier 0 is __syncthreads).
__device__ __forceinline__ void row_sync(int u, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(u + 1), "r"(n) : "memory");
}

template <int P>
struct SymArgs {
    const double *jrec;   // [3(P+1)][ld]
    const double *m;      // [ld]
    int64_t ld;           // row stride (the padded body count, a multiple of kSymR)
    int64_t N;            // bodies; positions N .. ld-1 are padding
    SymSched sc;
    double eps2, G;
    double *part;         // [2C][(P+1)*3][ld]
    unsigned long long *wmax;   // kH: max over pairs of G (m_i + m_j) s^(-3/2) (bit pattern), raised
};

// Record of body b.  Padding bodies get mass 0 and distinct far-away positions,
// so that no pair has r = 0 (their own sums are never read).
template <int P>
__device__ __forceinline__ void load_body(const SymArgs<P> &a, int64_t b, double (&r)[P + 1][3], double &gm)
{
    if (b < a.N) {
#pragma unroll
        for (int k = 0; k <= P; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) r[k][c] = a.jrec[(3 * k + c) * a.ld + b];
        gm = a.G * a.m[b];
    } else {
#pragma unroll
        for (int k = 0; k <= P; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) r[k][c] = 0.0;
        r[0][0] = kFarAway + (double)(b - a.N);
        gm = 0.0;
    }
}

template <int P>
__device__ __forceinline__ void rotate(double (&r)[P + 1][3], double &gm, int src)
{
#pragma unroll
    for (int k = 0; k <= P; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) r[k][c] = __shfl_sync(0xffffffffu, r[k][c], src);
    gm = __shfl_sync(0xffffffffu, gm, src);
}

// Subtiles [t0, t1) of the diagonal block of row I in FP64: ordered pairs into the
// i-side sums only.  kH: a padding body counts for no pair, however close it is.
template <int P, bool kH>
__device__ __forceinline__ void ring_diag(const SymArgs<P> &a, int I, int t0, int t1, int w, int lane,
                                          const double (&ri)[P + 1][3], double gmi, double (&acci)[P + 1][3],
                                          unsigned long long &wm)
{
    const int src = (lane + 1) & 31;
    for (int js = t0; js < t1; ++js) {
        double rj[P + 1][3], gmj;
        load_body<P>(a, (int64_t)I * kSymR + js * 32 + lane, rj, gmj);
        [[maybe_unused]] const int64_t n_real =
            (int64_t)I * kSymR + w * 32 + lane < a.N ? a.N - ((int64_t)I * kSymR + js * 32) : 0;
        for (int t = 0; t < 32; ++t) {
            const bool self = js == w && t == 0;
            double r[P + 1][3];
#pragma unroll
            for (int k = 0; k <= P; ++k)
#pragma unroll
                for (int c = 0; c < 3; ++c) r[k][c] = rj[k][c] - ri[k][c];
            double s = fma(r[0][0], r[0][0], fma(r[0][1], r[0][1], fma(r[0][2], r[0][2], a.eps2)));
            s = self ? 1.0 : s;
            const double wi = self ? 0.0 : gmj;
            const double rinv = rsqrt_fp64(s);
            const double sinv = rinv * rinv;
            const double S = rinv * sinv;
            const double mS = wi * S;
            if constexpr (kH) {
                const bool real = !self && ((lane + t) & 31) < n_real;
                const unsigned long long wb = real ? (unsigned long long)__double_as_longlong((gmi + gmj) * S) : 0ull;
                wm = wb > wm ? wb : wm;
            }
            pair_odd_terms<P, double>(r, sinv, [&](int k, int c, double B) {
                acci[k][c] = fma(mS, B, acci[k][c]);
            });
            rotate<P>(rj, gmj, src);
        }
    }
}

// One 32-body j-subtile (bodies jb .. jb + 31) against the warp's i-bodies in
// FP64: a ring in which the j-body and its j-side sums accj travel lane by lane.
// real_i: this thread's i-body is no padding.
template <int P, bool kH>
__device__ __forceinline__ void ring_tile(const SymArgs<P> &a, int64_t jb, int lane, bool real_i,
                                          const double (&ri)[P + 1][3], double gmi, double (&acci)[P + 1][3],
                                          double (&accj)[P + 1][3], unsigned long long &wm)
{
    [[maybe_unused]] const int64_t n_real = real_i ? a.N - jb : 0;      // j-lanes that hold bodies
    const int src = (lane + 1) & 31;      // after t passes lane l holds j-lane (l + t) mod 32
    double rj[P + 1][3], gmj;
    load_body<P>(a, jb + lane, rj, gmj);
    for (int t = 0; t < 32; ++t) {
        double r[P + 1][3];
#pragma unroll
        for (int k = 0; k <= P; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) r[k][c] = rj[k][c] - ri[k][c];
        const double s = fma(r[0][0], r[0][0], fma(r[0][1], r[0][1], fma(r[0][2], r[0][2], a.eps2)));
        const double rinv = rsqrt_fp64(s);
        const double sinv = rinv * rinv;
        const double S = rinv * sinv;
        const double wi = gmj * S, wj = gmi * S;
        if constexpr (kH) {
            const unsigned long long wb =
                ((lane + t) & 31) < n_real ? (unsigned long long)__double_as_longlong(wi + wj) : 0ull;
            wm = wb > wm ? wb : wm;
        }
        pair_odd_terms<P, double>(r, sinv, [&](int k, int c, double B) {
            acci[k][c] = fma(wi, B, acci[k][c]);
            accj[k][c] = fma(-wj, B, accj[k][c]);
        });
        rotate<P>(rj, gmj, src);
#pragma unroll
        for (int k = 0; k <= P; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) accj[k][c] = __shfl_sync(0xffffffffu, accj[k][c], src);
    }
}

// Launch configuration: a plan with one item per CTA is launched cooperatively,
// so that the runtime makes all its CTAs resident at once (its turns wait on
// CTAs of the same launch in any order); otherwise a plain launch.
struct SymLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    SymLaunch(const SymLaunch &) = delete;
    SymLaunch(const SymPlan &pl, int threads, cudaStream_t st)
    {
        cfg.gridDim = dim3((unsigned)pl.grid);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = pl.cyclic ? 1 : 0;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

inline SymSched make_sched(const SymPlan &pl, const SymSync &sy)
{
    return SymSched{pl.nB, pl.D, pl.C, pl.Bc, pl.H, pl.G, pl.K, pl.cyclic ? 1 : 0, pl.items, sy.words, sy.words + 1,
                    sy.flag, sy.wait_ns, sy.bias};
}

}  // namespace mh
