// sweep_block.cuh -- the sweep of QUIO models whose dependency levels are
// narrow (complete and nearly complete graphs, where every level holds one
// variable or a few), in blocks of 32 consecutive variables.
//
// One warp of the replica's group decides a block: lane i holds variable
// kb + i, its field f and its random words in registers.  All undecided lanes
// decide at once from the present fields.  A decision is final when no earlier
// lane of the block that shares a term with it changes in the same round, since
// everything before it in the visiting order is then already in its field; the
// leading final lanes commit, their changes go into the fields of the other
// lanes (the 32 x 32 couplings of the block, DevModel::blk_w), and the rest
// decide again.  The sequential order of Sect. 3.1 is kept exactly, changes are
// added to a field in that order, and nothing but warp shuffles separates two
// changes of a block.  Changes reach the other fields block by block.
//
// What bounds it: the chain of rounds (decision, two ballots, one coupling row
// from shared memory).  Deciding level by level, or a window of
// levels up to its first change, cost two group barriers, a Philox block and an
// L2 row per change instead (about 2500 cycles).
#pragma once

namespace sa {
namespace dev {

// What a thread carries through the sweeps of a run.
template <class F>
struct SweepAcc {
    typename Num<F>::Acc e;          // energy share
    unsigned long long changes;
    float de;                        // float models: energy changes since the last fold into e
    float drift;                     // float models: largest error of a field seen by a refresh
    int busy;                        // heat bath: changes of the last block
    int turn;                        // blocks begun: which staged place is current
    int par;                         // blocked sweeps: which of the two commit lists is current
    int last;                        // and the block whose changes are not applied everywhere yet (-1: none)
};

// Heat bath over narrow ranges: a round of lane decisions settles 1 / p
// variables when a share p of them changes and costs about 2700 cycles (16
// values: one warp issues an instruction every four to five cycles, and the
// lanes' loops have some 500); in turn, with a variable's values spread over the
// lanes, it is about 600 a variable.  Above this many changes in the last block
// they go in turn (the results are the same).  Complete graphs of 32 and 200
// variables over 4 to 32 values, 64 and 1024 replicas: a limit of 3 costs up to 9%
// more (6% less for int64 over 4 values, 200 variables), one of 12 from 8% less
// (fp32) to 11% more (int64, 200 variables, 32 values: 4.72 -> 5.25 ms).
constexpr int kBusyBlock = 6;

// A change of the block: {variable, z_new - z_old, first entry and length of its row}.
using Commit = int4;

// ------------------------------------------------------------------ heat bath, one variable per warp
// heat_bath_general of a QUIO variable, evaluated by a warp with the same
// additions in the same order (the pick is bit for bit the same): the weights
// come from the lanes, the compensated sum is one chain that every lane
// follows, and the sums after each value -- the second pass of the scalar form
// repeats them -- stay in the lanes, where a ballot finds the pick.  At most
// kChainValues values.
constexpr uint32_t kChainValues = 192;

template <class F>
__device__ __forceinline__ long long heat_bath_chain(const VarView<F, KIND_QUIO>& vv, long long z, long long lo,
                                                     uint32_t width, uint32_t xu, float beta, int lane) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int H = kChainValues / 32;
    F mn = F(0);
    const F e = quio_interval_min<F>(vv, z, lo, lo + (long long)width);
    mn = e < mn ? e : mn;
    uint32_t wb0 = 0, wb1 = width / 32;
    // (a single block of 32 values is kept whatever the window says)
    if (wb1 > 0) hb_quio_window<F>(vv, z, lo, width, mn, beta, wb0, wb1);
    const uint32_t c0 = wb0 * 32, c1 = min(width, wb1 * 32 + 31);
    const float zf = __int2float_rn((int)z), v0f = __int2float_rn((int)lo);
    const float b2 = beta * 1.4426950408889634f, mb = Num<F>::to_f(mn) * b2;
    const int n = (int)(c1 - c0) + 1;
    // the scalar form reaches a value by steps of 1 from its block of 32; beyond
    // 2^24 the steps round
    const bool steps_round = Num<F>::is_float && !(fabsf(v0f) + (float)width < 16777216.f);
    float pre[H];
    float sum = 0.f, comp = 0.f;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        pre[h] = 0.f;
        if (32 * h < n) {
            const uint32_t i0 = c0 + (uint32_t)(32 * h + lane);
            float w = 0.f;
            if (i0 <= c1) {
                if constexpr (Num<F>::is_float) {
                    float vf = v0f + (float)i0;
                    if (steps_round) {
                        vf = v0f + (float)(c0 + 32u * h);
                        for (int i = 0; i < lane; ++i) vf += 1.f;
                    }
                    w = ex2_ftz(fmaf(-vv.delta_ff(zf, vf), b2, mb));
                } else w = expf(-(Num<F>::to_f(vv.delta(z, lo + (long long)i0) - mn) * beta));
            }
            const int cnt = min(32, n - 32 * h);
#pragma unroll 4
            for (int i = 0; i < cnt; ++i) {
                const float y = __shfl_sync(full, w, i) - comp;
                const float t = sum + y;
                comp = (t - sum) - y;
                sum = t;
                if (lane == i) pre[h] = sum;
            }
        }
    }
    const float thr = unit_open_left(xu) * sum;
    int pick = n - 1;
#pragma unroll
    for (int h = H - 1; h >= 0; --h) {
        const unsigned hit = __ballot_sync(full, 32 * h + lane < n && pre[h] >= thr);
        if (hit) pick = 32 * h + __ffs(hit) - 1;
    }
    return lo + (long long)(c0 + (uint32_t)pick);
}

// heat_bath_quio_f32_small evaluated by a warp, with the same additions in the
// same order: two blocks of 16 values at a time (a half warp each, the tree of
// the scalar form as four exchanges), the block sums' chain in every lane.
__device__ __forceinline__ long long heat_bath_small_warp(float f, float d, long long z, long long lo, uint32_t width,
                                                          uint32_t xu, float beta, float temp, int lane) {
    constexpr unsigned full = 0xffffffffu;
    const HbWindow q = hb_small_window(f, d, z, lo, width, beta, temp);
    const int j = lane & 15;
    float run = 0.f, pre = 0.f;   // sum of the blocks so far; lane b: the sum up to and with block b
#pragma unroll 2
    for (int b = 0; b < q.nrb; b += 2) {
        const int mb = b + (lane >> 4);   // this half warp's block
        const int cnt = min(16, q.n - (q.base + mb * 16));
        float w = 0.f;
        if (mb < q.nrb && j < cnt) w = quio_w((q.dzb0 + (float)(mb * 16)) + (float)j, q.hA, q.hB, q.mb);
        float tree = w;
#pragma unroll
        for (int h = 8; h >= 1; h >>= 1) tree += __shfl_xor_sync(full, tree, h);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (b + s >= q.nrb) break;
            const int c = min(16, q.n - (q.base + (b + s) * 16));
            float acc;
            if (c == 16) {
                acc = __shfl_sync(full, tree, 16 * s);
            } else {   // the range's last, partial block: summed in order
                acc = 0.f;
                for (int i = 0; i < c; ++i) acc += __shfl_sync(full, w, 16 * s + i);
            }
            run += acc;
            if (lane == b + s) pre = run;
        }
    }
    const float thr = unit_open_left(xu) * run;
    const unsigned hit = __ballot_sync(full, lane < q.nrb && pre >= thr);
    // rounding can leave the threshold above the window: its last block
    const int sel = hit ? __ffs(hit) - 1 : q.nrb - 1;
    run = sel > 0 ? __shfl_sync(full, pre, sel - 1) : 0.f;
    const int first = q.base + sel * 16;
    const int cnt = min(16, q.n - first);
    const float w = j < cnt ? quio_w((q.dz0 + (float)first) + (float)j, q.hA, q.hB, q.mb) : 0.f;
    float mine = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        run += __shfl_sync(full, w, i);
        if (j == i) mine = run;
    }
    const unsigned h2 = __ballot_sync(full, j < cnt && mine >= thr) & 0xffffu;
    return lo + (long long)(first + (h2 ? __ffs(h2) - 1 : cnt - 1));
}

// heat_bath_chain where the range has at most 32 values and the numbers are
// small (see heat_bath_narrow): 32-bit arithmetic, the minimum by one warp
// reduction.
__device__ __forceinline__ int heat_bath_chain32(int f, int d, int z, int lo, uint32_t width, uint32_t xu, float beta,
                                                 int lane) {
    constexpr unsigned full = 0xffffffffu;
    const int v = lo + lane;
    const bool in = (uint32_t)lane <= width;
    const int de = (v - z) * (f + d * (v + z));
    const int mn = __reduce_min_sync(full, in ? de : 0);   // (0, at z, is among them)
    const float w = expf(-(__int2float_rn(de - mn) * beta));
    float sum = 0.f, comp = 0.f, pre = 0.f;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        if (8u * g > width) break;   // the same for every lane
        float wi[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) wi[j] = __shfl_sync(full, w, 8 * g + j);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // (values past the range come last and are never looked at)
            const float y = wi[j] - comp;
            const float t = sum + y;
            const bool ok = (uint32_t)(8 * g + j) <= width;
            comp = ok ? (t - sum) - y : comp;
            sum = ok ? t : sum;
            pre = lane == 8 * g + j ? sum : pre;
        }
    }
    const float thr = unit_open_left(xu) * sum;
    const unsigned hit = __ballot_sync(full, in && pre >= thr);
    return lo + (hit ? __ffs(hit) - 1 : (int)width);
}
__device__ __forceinline__ bool small_numbers(long long f, long long d, int lo, uint32_t width) {
    return width < 32u && f < (1 << 23) && f > -(1 << 23) && d < (1 << 10) && d > -(1 << 10) && lo > -(1 << 12) &&
           (long long)lo + (long long)width < (1 << 12);
}

// One variable's heat-bath draw by a whole warp (out of line: four forms that
// would each hold registers of the block loop).
template <class F>
__device__ __noinline__ int heat_bath_in_turn(F f, F d, int z, int lo, uint32_t width, uint32_t xu, float beta,
                                              float temp, int lane, bool wide) {
    VarView<F, KIND_QUIO> vv;
    vv.f = f;
    vv.d = d;
    if (vv.linear()) return (int)heat_bath_linear(Num<F>::to_f(f), lo, width, xu, beta);
    if constexpr (!Num<F>::is_float)
        if (!wide && small_numbers(f, d, lo, width))
            return heat_bath_chain32((int)f, (int)d, z, lo, width, xu, beta, lane);
    if (wide) return (int)heat_bath_warp<F, KIND_QUIO>(vv, z, lo, width, xu, beta, lane);
    if (Num<F>::is_float && width < 256u && lo > -(1 << 22) && (long long)lo + (long long)width < (1 << 22))
        return (int)heat_bath_small_warp((float)f, (float)d, z, lo, width, xu, beta, temp, lane);
    if (width < kChainValues) return (int)heat_bath_chain<F>(vv, z, lo, width, xu, beta, lane);
    return (int)heat_bath_general<F, KIND_QUIO>(vv, z, lo, width, xu, beta);
}

// A lane's own variable, narrow range (out of line for the same reason).
template <class F>
__device__ __noinline__ int heat_bath_lane(F f, F d, int z, int lo, uint32_t width, uint32_t xu, float beta, float temp,
                                           uint32_t max_width) {
    VarView<F, KIND_QUIO> vv;
    vv.f = f;
    vv.d = d;
    if (vv.linear()) return (int)heat_bath_linear(Num<F>::to_f(f), lo, width, xu, beta);
    if constexpr (Num<F>::is_float) {
        if (lo > -(1 << 22) && (long long)lo + (long long)width < (1 << 22))
            return (int)heat_bath_quio_f32_small((float)f, (float)d, z, lo, width, xu, beta, temp);
        return (int)heat_bath_general<F, KIND_QUIO>(vv, z, lo, width, xu, beta);
    } else {
        return (int)heat_bath_narrow(vv, z, lo, width, xu, beta, max_width);
    }
}

// ------------------------------------------------------------------ changes to the other fields
// Fields of a complete graph: the commits' couplings to field j, in order.  Row
// k lists every j != k in order, so entry j - [j > k] of the row is J_kj.  Rows
// are read past L1 (each entry is used once), NR at a time and for NF fields at a
// time, all loads before the first addition.
// (Predicates instead of branches throughout: a uniform branch per row costs
// more than the row.)
template <class F, int NF, int NR>
struct RowPart {
    F w[NF][NR];
    int dz[NR];          // 0 beyond the last commit
};
template <class F, int NF, int NR>
__device__ __forceinline__ void load_rows(RowPart<F, NF, NR>& q, const DevModel& m, const Commit* list, int c, int count,
                                          const int (&j)[NF]) {
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const Commit e = list[(c + u) & 31];   // (entries beyond the count are read and not used)
        const bool on = c + u < count;
        q.dz[u] = on ? e.y : 0;
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            q.w[i][u] = F(0);
            if (on && j[i] >= 0) q.w[i][u] = Coef<F>::adj_once(m, e.z + j[i] - (j[i] > e.x ? 1 : 0));
        }
    }
}
template <class F, int NF, int NR>
__device__ __forceinline__ void add_rows(const RowPart<F, NF, NR>& q, F (&f)[NF]) {
#pragma unroll
    for (int u = 0; u < NR; ++u)
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            F g = f[i];
            solo_add(&g, q.w[i][u], q.dz[u]);
            f[i] = q.dz[u] != 0 ? g : f[i];
        }
}
// Every field outside of blocks b0 and b1, by threads t = 0..nt-1: four fields
// (two for int64) with eight (four) rows each in flight per thread.  A pass is
// one L2 round trip, about 1700 cycles when every SM reads rows: with two fields
// at a time the 1000-variable case below took 6.8 ms instead of 6.4.
template <class F, int MEM>
__device__ __noinline__ void add_commits(const DevModel& m, F* cache_any, const Commit* list_any, int count, int b0,
                                         int b1, int t, int nt) {
    constexpr int NF = Num<F>::is_float ? 4 : 2, NR = Num<F>::is_float ? 8 : 4;
    F* cache = in_shared<MEM>(cache_any);
    const Commit* list = in_shared<MEM>(list_any);
    const int n = m.n;
    for (int j0 = t; j0 < n; j0 += NF * nt) {
        int j[NF];
        F f[NF];
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            j[i] = j0 + i * nt;
            if (j[i] >= n || (j[i] >> 5) == b0 || (j[i] >> 5) == b1) j[i] = -1;
            f[i] = j[i] >= 0 ? cache[j[i]] : F(0);
        }
        for (int c = 0; c < count; c += NR) {
            RowPart<F, NF, NR> q;
            load_rows<F, NF, NR>(q, m, list, c, count, j);
            add_rows<F, NF, NR>(q, f);
        }
#pragma unroll
        for (int i = 0; i < NF; ++i)
            if (j[i] >= 0) cache[j[i]] = f[i];
    }
}

// The commits' rows by columns, integer fields of any graph: every thread of `nt`
// takes the next (commit, link) pair.  Columns of block `own` already have the change.
template <class F, int MEM>
__device__ __noinline__ void scatter_commits(const DevModel& m, F* cache_any, const Commit* list_any, int count, int own,
                                             int t, int nt) {
    F* cache = in_shared<MEM>(cache_any);
    const Commit* list = in_shared<MEM>(list_any);
    const int lane = t & 31;
    const int len = lane < count ? list[lane].w : 0;
    int inc = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    const int W = __shfl_sync(0xffffffffu, inc, 31);
    auto find = [&](int w, int& dz) -> int {
        int h = 0;   // number of commits whose rows end at or before w
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, inc, h + o - 1) <= w) h += o;
        const int pre = __shfl_sync(0xffffffffu, inc - len, h);
        if (w >= W) return -1;
        const Commit e = list[h];
        dz = e.y;
        return e.z + (w - pre);
    };
    for (int w0 = t - lane; w0 < W; w0 += 2 * nt) {
        int dz[2] = {0, 0}, at[2], col[2];
        F wt[2];
        at[0] = find(w0 + lane, dz[0]);
        at[1] = w0 + nt < W ? find(w0 + nt + lane, dz[1]) : -1;
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (at[u] >= 0) {
                col[u] = __ldg(m.adj_col + at[u]);
                wt[u] = Coef<F>::adj(m, at[u]);
            }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (at[u] >= 0 && (col[u] >> 5) != own) atomic_add_field<MEM>(cache + col[u], wt[u] * (F)dz[u]);
    }
}

// fp32 fields of any graph: every field takes its changes in the order of the
// commits, so that a run's results do not depend on its threads.  Each of `nw`
// warps (a power of two) owns a range of columns and walks the commits over its
// part of their rows (rows are sorted by column, DevModel::blk_part holds where the
// parts begin), 32 links at a time with plain reads and writes; eight such pieces
// are loaded before the first is added.
// What bounds it: the instructions of a piece (about 25) and its shared-memory
// round trip, one warp's chain; sixteen pieces at a time or the next eight loaded
// ahead cost more in pieces past the last.  1000 variables, Metropolis, 64 / 1024
// replicas x 20 sweeps, unordered atomics over all threads against this: rows of 40
// links 2.01 / 3.45 ms against 2.26 / 3.17, 120 links 2.26 / 6.65 against 2.55 /
// 5.17, 500 links 4.54 / 22.5 against 4.26 / 15.0.
template <int MEM>
__device__ __noinline__ void ordered_commits(const DevModel& m, float* cache_any, const Commit* list_any, int count,
                                             int own, int warp, int nw, int lane) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int U = 8;
    float* cache = in_shared<MEM>(cache_any);
    const Commit* list = in_shared<MEM>(list_any);
    // lane c: commit c's part of this warp's columns
    int first = 0, last = 0;
    if (lane < count) {
        const Commit e = list[lane];
        last = e.w;
        if (nw > 1) {
            const int* part = m.blk_part + (size_t)e.x * kRowParts + warp * (kRowParts / nw);
            first = __ldg(part);
            if (warp + 1 < nw) last = __ldg(part + kRowParts / nw);
        }
    }
    const int pieces = (last - first + 31) >> 5;
    int upto = pieces;   // pieces of commits 0..lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(full, upto, o);
        if (lane >= o) upto += u;
    }
    const int total = __shfl_sync(full, upto, 31);
    const int start = first - 32 * (upto - pieces);   // piece i, if it is commit lane's, begins 32 i later
    // (no branches: past the last piece the commit is the first one and `at` lies
    // beyond its part)
    for (int i0 = 0; i0 < total; i0 += U) {
        int col[U];
        float inc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int h = __popc(__ballot_sync(full, upto <= i0 + u)) & 31;   // the piece's commit
            const Commit e = list[h];
            const int at = __shfl_sync(full, start, h) + 32 * (i0 + u) + lane;
            const bool on = at < __shfl_sync(full, last, h);
            col[u] = 32 * own;
            inc[u] = 0.f;
            if (on) col[u] = __ldg(m.adj_col + e.z + at);
            if (on) inc[u] = __fmul_rn(Coef<float>::adj(m, e.z + at), (float)e.y);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if ((col[u] >> 5) != own) cache[col[u]] = __fadd_rn(cache[col[u]], inc[u]);
            __syncwarp();   // a column may come again in the next commit
        }
    }
}

// Integer rows with fewer links than this in all are scattered by the deciding
// warp (1000 variables of 40 links, 64 replicas x 40 sweeps: 32 links 3.89 ms, 96
// 3.97, 300 4.36; 320 of 20: 1.19, 1.18, 1.25), and fp32 rows with fewer pieces
// than this beyond one per commit (320 variables of 30 links, 64 replicas: 16
// pieces 0.89 ms, 6 0.86; 2 is as good as 6).
constexpr int kScatterAlone = 96;
constexpr int kPiecesAlone = 6;

// The commits' rows by the `nt` threads t = 0..nt-1.
template <class F, int MEM>
__device__ __forceinline__ void group_scatter(const DevModel& m, F* cache, const Commit* list, int count, int own, int t,
                                              int nt) {
    if constexpr (Num<F>::is_float) {
        // a power of two of warps, as many as the longest row has pieces
        int nw = 1;
        if (nt > 32) {
            const int lane = t & 31;
            const int longest = __reduce_max_sync(0xffffffffu, lane < count ? list[lane].w : 0);
            while (nw < kRowParts && 2 * nw <= (nt >> 5) && 32 * nw < longest) nw *= 2;
            if ((t >> 5) >= nw) return;
        }
        ordered_commits<MEM>(m, cache, list, count, own, t >> 5, nw, t & 31);
    } else {
        scatter_commits<F, MEM>(m, cache, list, count, own, t, nt);
    }
}

// ------------------------------------------------------------------ one block
// Block b's couplings, records and masks on their way into one of the two
// staged places (asynchronous 16-byte copies, issued one block ahead: an
// L1 prefetch of the same lines left every coupling row an L2 round trip, about
// 600 cycles a round).  Places lie behind state regions in shared memory alone.
template <int MEM>
__device__ __forceinline__ bool blocks_staged(const SweepArgs& a) {
    return MEM != MEM_GLOBAL && a.off_blk >= 0;
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void stage_block(const DevModel& m, uint8_t* place, int b, int lane, bool records) {
    const int4* w = reinterpret_cast<const int4*>(m.blk_w + (size_t)b * 1024);
    const int4* rec = reinterpret_cast<const int4*>(m.idx_rec + b * 32);
    const int recs = records ? min(32, m.n - b * 32) : 0;
    int4* dw = reinterpret_cast<int4*>(place);
    int4* dr = reinterpret_cast<int4*>(place + 4096);
    uint32_t* dm = reinterpret_cast<uint32_t*>(place + 4096 + 32 * sizeof(LevelRec));
#pragma unroll
    for (int i = 0; i < 8; ++i) cp_async16(dw + 32 * i + lane, w + 32 * i + lane);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (32 * i + lane < 2 * recs) cp_async16(dr + 32 * i + lane, rec + 32 * i + lane);
    if (lane < recs) cp_async4(dm + lane, m.blk_mask + b * 32 + lane);
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A lane's variable: what its decisions need besides the field.
template <class F>
struct BlockLane {
    int k, lo, row, len;
    uint32_t width;      // 0 beyond the last variable
    unsigned nbr;        // earlier lanes of the block that share a term with this one
    int lvl;             // width of its dependency level
    uint32_t zo;
    F d;
    Words4 x;
    long long z, prop;   // prop: the proposed value where it does not depend on the field
    bool opt;            // optimal-transition proposal
};

// Block b's records, random words and proposals: nothing here waits for the
// changes of earlier blocks.
template <class F, class Z, int RULE>
__device__ __forceinline__ BlockLane<F> block_lane(const SweepArgs& a, const Z* zs, const uint8_t* place, bool staged,
                                                   int b, int s, int r, int lane) {
    const DevModel& m = a.m;
    BlockLane<F> q;
    q.k = b * 32 + lane;
    int4 x0 = make_int4(0, 0, 0, 0), x1 = x0;
    q.nbr = 0;
    q.zo = 0;
    if (q.k < m.n) {
        if (staged) {
            const int4* p = reinterpret_cast<const int4*>(place + 4096) + 2 * lane;
            x0 = p[0];
            x1 = p[1];
            q.nbr = reinterpret_cast<const uint32_t*>(place + 4096 + 32 * sizeof(LevelRec))[lane];
        } else {
            const int4* p = reinterpret_cast<const int4*>(m.idx_rec + q.k);
            x0 = __ldg(p);
            x1 = __ldg(p + 1);
            q.nbr = __ldg(m.blk_mask + q.k);
        }
        q.zo = (uint32_t)zs[q.k];
    }
    q.lo = x0.y;
    q.width = (uint32_t)x0.z;
    q.row = x0.w;
    q.len = x1.x;
    q.lvl = x1.y;
    if constexpr (Num<F>::is_float) q.d = __uint_as_float((uint32_t)x1.z);
    else q.d = (long long)(((unsigned long long)(uint32_t)x1.w << 32) | (uint32_t)x1.z);
    q.x = philox4x32_10((uint32_t)q.k, (uint32_t)s, (uint32_t)r, a.inst, a.key0, a.key1);
    q.z = (long long)q.lo + (long long)q.zo;
    q.prop = q.z;
    q.opt = false;
    if (RULE != RULE_HEAT_BATH && q.width != 0u) {
        if (RULE == RULE_OPT) q.opt = unit_open_right(q.x.x2) < __ldg(a.ratio + s);
        if (!q.opt) {
            const uint32_t j = pick_below(q.x.x0, q.width);
            q.prop = (long long)q.lo + (long long)(j >= q.zo ? j + 1u : j);
        }
    }
    return q;
}

// Energy changes of a sweep: where every level holds one variable one lane sums
// them in the visiting order, which is the level order's sum; elsewhere every lane
// sums its own variables' changes, as the threads of a level do (one fp32 sum of
// a sweep's changes had four to nine times the rounding error for levels of 5 to 16).
template <class F>
__device__ __forceinline__ bool sum_in_order(const DevModel& m) {
    return Num<F>::is_float && m.n_levels == m.n;
}

// Decides block b (warp-collective) from the lanes' fields; on return f holds
// every change of the block, the list its commits.  Returns their number.
// `dense` (a constant at each call): a complete graph.
template <class F, class Z, int RULE, int MEM>
__device__ __forceinline__ int decide_block(const SweepArgs& a, const BlockLane<F>& q, const uint8_t* place, Z* zs, F& f,
                                            Commit* list, int b, int s, int r, float beta, float temp, int lane,
                                            SweepAcc<F>& acc, const bool dense) {
    constexpr unsigned full = 0xffffffffu;
    const DevModel& m = a.m;
    // row p of the block's couplings
    const int* const blk = reinterpret_cast<const int*>(place) + lane;
    const bool staged = blocks_staged<MEM>(a), in_order = dense ? Num<F>::is_float : sum_in_order<F>(m);
    auto coupling = [&](int p) -> F {
        const size_t at = (size_t)b * 1024 + 32 * p + lane;
        const int w = staged ? blk[32 * p] : __ldg(m.blk_w + at);
        if constexpr (Num<F>::is_float) return __int_as_float(w);
        else return m.blk_i == nullptr ? (long long)w : (long long)__ldg(m.blk_i + at);
    };
    const long long z = q.z;
    long long v = z;
    int count = 0;
    // heat bath: narrow ranges are decided by the lanes (rounds, like the other
    // rules) unless most of the last block changed; other ranges one variable
    // after the other by the whole warp
    bool in_turn = false;
    if constexpr (RULE == RULE_HEAT_BATH)
        in_turn = m.max_width >= (Num<F>::is_float ? 64u : 32u) || acc.busy > kBusyBlock;
    if (RULE == RULE_HEAT_BATH && in_turn) {
        // the scalar or the warp-wide sum, whichever the level order takes for
        // the variable's level (the sums differ in their last bits)
        const unsigned wide = __ballot_sync(full, hb_warp_mode(q.lvl, a.hb_tpr, m.max_width,
                                                               Num<F>::is_float && m.max_width < 256u));
        unsigned left = __ballot_sync(full, q.width != 0u);
        while (left) {
            const int p = __ffs(left) - 1;
            left &= left - 1u;
            const F w = coupling(p);
            VarView<F, KIND_QUIO> vv;
            vv.f = __shfl_sync(full, f, p);
            vv.d = __shfl_sync(full, q.d, p);
            const uint32_t wp = __shfl_sync(full, q.width, p);
            const int lp = __shfl_sync(full, q.lo, p);
            const int zp = lp + (int)__shfl_sync(full, q.zo, p);
            const int vp = heat_bath_in_turn<F>(vv.f, vv.d, zp, lp, wp, __shfl_sync(full, q.x.x0, p), beta, temp, lane,
                                                (wide >> p) & 1u);
            if (vp != zp) {
                const int dz = vp - zp;
                if (in_order ? lane == 0 : lane == p) {
                    const F dp = vv.delta(zp, vp);
                    if constexpr (Num<F>::is_float) acc.de = __fadd_rn(acc.de, (float)dp);   // (no fused multiply-add)
                    else acc.e += dp;
                }
                if (lane == p) {
                    v = vp;
                    list[count] = make_int4(q.k, dz, q.row, q.len);
                    zs[q.k] = (Z)(vp - lp);
                    ++acc.changes;
                } else {
                    solo_add(&f, w, dz);
                }
                ++count;
            }
        }
    } else {
        // A round keeps to one path for all lanes and writes nothing: the list,
        // the state and the energy follow when the block is decided.
        unsigned open = __ballot_sync(full, q.width != 0u), changed = 0u;   // lanes still to be decided, changed
        const float u = unit_open_right(q.x.x1);
        // the proposal's share of dE = (v - z) (f + J_kk (v + z)) (quio_delta)
        int dz = 0, dz_done = 0;
        F dv = F(0), sv = F(0), de = F(0);
        auto propose = [&](long long pv) {
            dz = (int)(pv - z);
            if constexpr (Num<F>::is_float) {
                const float vf = __int2float_rn((int)pv), zf = __int2float_rn((int)z);
                dv = vf - zf;
                sv = vf + zf;
            } else {
                dv = pv - z;
                sv = q.d * (pv + z);
            }
        };
        propose(q.prop);
        while (open) {
            const bool mine = (open >> lane) & 1u;
            if constexpr (RULE == RULE_HEAT_BATH) {
                if (mine) propose(heat_bath_lane<F>(f, q.d, (int)z, q.lo, q.width, q.x.x0, beta, temp, m.max_width));
            } else if constexpr (RULE == RULE_OPT) {
                if (mine && q.opt) {
                    VarView<F, KIND_QUIO> vv;
                    vv.f = f;
                    vv.d = q.d;
                    propose(opt_argmin<F, KIND_QUIO>(vv, z, q.lo, (long long)q.lo + (long long)q.width));
                }
            }
            F dn;
            if constexpr (Num<F>::is_float) dn = __fmul_rn(dv, fmaf(q.d, sv, f));
            else dn = dv * (f + sv);
            bool chg = mine & (dz != 0);
            if (RULE != RULE_HEAT_BATH) {   // metropolis_accept without its branch
                const float pr = expf(-(Num<F>::to_f(dn) * beta));
                chg = chg & ((dn <= F(0)) | (u < pr));
            }
            const unsigned c = __ballot_sync(full, chg);
            if (!c) break;
            // the first lane whose field one of the changes reaches decides
            // again; on a complete graph that is the next lane
            unsigned done;
            if (dense) {
                const unsigned low = c & (0u - c);
                done = low | (low - 1u);
            } else {
                const unsigned late = __ballot_sync(full, mine && (q.nbr & c) != 0u);
                done = late ? (late & (0u - late)) - 1u : full;
            }
            unsigned com = c & done;
            changed |= com;
            open &= ~done;
            const bool now = (com >> lane) & 1u;
            dz_done = now ? dz : dz_done;
            de = now ? dn : de;
            do {
                const int p = __ffs(com) - 1;
                com &= com - 1u;
                F g = f;
                solo_add(&g, coupling(p), __shfl_sync(full, dz, p));
                f = lane != p ? g : f;
            } while (com);
        }
        count = __popc(changed);
        v = z + dz_done;
        if ((changed >> lane) & 1u) {
            list[__popc(changed & ((1u << lane) - 1u))] = make_int4(q.k, dz_done, q.row, q.len);
            zs[q.k] = (Z)(v - (long long)q.lo);
            ++acc.changes;
            if constexpr (!Num<F>::is_float) acc.e += de;
            else if (!in_order) acc.de = __fadd_rn(acc.de, (float)de);
        }
        if constexpr (Num<F>::is_float) {   // else by one lane, four at a time
            for (unsigned c = in_order ? changed : 0u; c;) {
                float ep[4];
                bool on[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    on[i] = c != 0u;
                    ep[i] = __shfl_sync(full, (float)de, __ffs(c | 0x80000000u) - 1);
                    c &= c - 1u;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) acc.de = on[i] && lane == 0 ? __fadd_rn(acc.de, ep[i]) : acc.de;
            }
        }
    }
    if constexpr (RULE == RULE_HEAT_BATH) acc.busy = count;
    if (a.trace != nullptr && r < a.trace_R && q.k < m.n)
        a.trace[((size_t)s * a.trace_R + r) * m.n + q.k] = (int32_t)v;
    return count;
}

// Whether two warps take the blocks of a complete graph in turn: the one that
// does not decide makes the next block's random words and proposals (they need
// no field) and fetches its couplings, so that the deciding warp only adds the
// last changes and runs its rounds.  Each warp has a staged place of its own.
__device__ __forceinline__ bool block_pair(int tpr, int nb) { return tpr >= 128 && nb >= 2; }
template <class F, class Z, int RULE, int MEM>
__device__ __forceinline__ void prepare_block(const SweepArgs& a, const Z* zs, uint8_t* place, int b, int s, int r,
                                              int lane, BlockLane<F>& q) {
    if (s >= a.S) return;
    if (blocks_staged<MEM>(a)) stage_block(a.m, place, b, lane, false);
    q = block_lane<F, Z, RULE>(a, zs, place, false, b, s, r, lane);
}

// ------------------------------------------------------------------ one sweep
// Sweep s of replica r in blocks.  `flush`: the caller needs the state at the
// end of this sweep (a refresh, a trace, the outputs), so the last block's
// changes are applied before returning; otherwise they wait for the next sweep.
//
// Complete graphs: while one warp decides block b, the others add the changes of
// block b - 1 to every field outside of blocks b - 1 and b (each field by one
// thread); the deciding warp adds them to block b's fields itself when it starts
// on them.  One barrier per block.
// Other graphs: warp 0 decides, then the group scatters the block's rows by
// their columns; short rows are scattered by warp 0 without waking the others.
// fp32 fields take their changes in the visiting order (see ordered_commits).
template <class F, class Z, int RULE, int MEM>
__device__ __forceinline__ void block_sweep(const SweepArgs& a, Z* zs, F* cache, int* ctl, Commit* lists, uint8_t* stage,
                                            int bar_id, int t, int tpr, int r, int s, bool flush, SweepAcc<F>& acc,
                                            BlockLane<F>& q) {
    const DevModel& m = a.m;
    const int lane = t & 31;
    const float beta = __ldg(a.beta + s);
    const float temp = 1.f / beta;
    const int nb = (m.n + 31) >> 5;
    // warp 0, at the start of block b: its staged place, with the next block's
    // copies issued (a model of one or two blocks stays staged), and its lanes
    auto begin = [&](int b) -> const uint8_t* {
        const bool staged = blocks_staged<MEM>(a);
        const uint8_t* place = stage + (nb > 2 ? (acc.turn & 1) : b) * kBlockStage;
        if (staged && nb > 2) {
            stage_wait();
            __syncwarp();   // every lane's copies of block b are there; block b - 1's place is free
            ++acc.turn;
            stage_block(m, stage + (acc.turn & 1) * kBlockStage, b + 1 < nb ? b + 1 : 0, lane, true);
        }
        q = block_lane<F, Z, RULE>(a, zs, place, staged, b, s, r, lane);
        return place;
    };
    if (m.dense_rows) {
        const bool pair = block_pair(tpr, nb);
        const int first = pair ? 64 : (tpr > 32 ? 32 : 0);   // first thread that only adds rows
        float* run = reinterpret_cast<float*>(ctl) + 8 + (s & 1);   // the sweep's energy change so far (float models)
        for (int b = 0; b < nb; ++b) {
            const Commit* prev = lists + 32 * (acc.par ^ 1);
            const int np = acc.last >= 0 ? ctl[acc.par ^ 1] : 0;
            if (pair ? (t >> 5) == acc.par : t < 32) {
                const int k = b * 32 + lane;
                const int ahead = acc.last != b ? np : 0;
                F f[1] = {k < m.n ? cache[k] : F(0)};
                const int j[1] = {k < m.n ? k : -1};
                constexpr int NR = 8;
                RowPart<F, 1, NR> ra, rb;
                load_rows<F, 1, NR>(ra, m, prev, 0, ahead, j);
                if (ahead > NR) load_rows<F, 1, NR>(rb, m, prev, NR, ahead, j);
                const uint8_t* place = stage + acc.par * kBlockStage;
                if (pair) {
                    stage_wait();
                    __syncwarp();
                    if (lane == 0) acc.de = b > 0 ? *run : 0.f;
                } else {
                    place = begin(b);
                }
                add_rows<F, 1, NR>(ra, f);
                if (ahead > NR) add_rows<F, 1, NR>(rb, f);
                for (int c = 2 * NR; c < ahead; c += NR) {
                    load_rows<F, 1, NR>(ra, m, prev, c, ahead, j);
                    add_rows<F, 1, NR>(ra, f);
                }
                const int cnt = decide_block<F, Z, RULE, MEM>(a, q, place, zs, f[0], lists + 32 * acc.par, b, s, r, beta,
                                                         temp, lane, acc, true);
                if (k < m.n) cache[k] = f[0];
                if (lane == 0) {
                    ctl[acc.par] = cnt;
                    if (pair) {
                        *run = acc.de;
                        acc.de = 0.f;
                    }
                }
            } else if (pair && t < 64) {
                prepare_block<F, Z, RULE, MEM>(a, zs, stage + (acc.par ^ 1) * kBlockStage, b + 1 < nb ? b + 1 : 0,
                                               b + 1 < nb ? s : s + 1, r, lane, q);
            }
            if (np > 0 && t >= first) add_commits<F, MEM>(m, cache, prev, np, acc.last, b, t - first, tpr - first);
            named_bar(bar_id, tpr);
            acc.par ^= 1;
            acc.last = b;
        }
        if (pair && t == 0) acc.de = *run;   // (read before the place's next use, two sweeps on)
        if (flush) {
            add_commits<F, MEM>(m, cache, lists + 32 * (acc.par ^ 1), ctl[acc.par ^ 1], acc.last, acc.last, t, tpr);
            named_bar(bar_id, tpr);
            acc.last = -1;
        }
    } else {
        // commands to the other warps: {commits or -1, their block}, in two
        // alternating places, so that one is read before it is written again
        if (t < 32) {
            for (int b = 0; b < nb; ++b) {
                const int k = b * 32 + lane;
                F f = k < m.n ? cache[k] : F(0);
                const uint8_t* place = begin(b);
                const int cnt = decide_block<F, Z, RULE, MEM>(a, q, place, zs, f, lists, b, s, r, beta, temp, lane, acc, false);
                if (k < m.n) cache[k] = f;
                __syncwarp();
                if (cnt == 0 || nb == 1) continue;
                bool together = false;
                if (tpr > 32) {
                    const int len = lane < cnt ? lists[lane].w : 0;
                    if constexpr (Num<F>::is_float)
                        together = __reduce_add_sync(0xffffffffu, (len + 31) >> 5) - cnt > kPiecesAlone;
                    else
                        together = __reduce_add_sync(0xffffffffu, len) > kScatterAlone;
                }
                if (together) {
                    if (lane == 0) {
                        ctl[4 + 2 * acc.par] = cnt;
                        ctl[5 + 2 * acc.par] = b;
                    }
                    acc.par ^= 1;
                    named_bar(bar_id, tpr);
                    group_scatter<F, MEM>(m, cache, lists, cnt, b, t, tpr);
                    named_bar(bar_id, tpr);
                } else {
                    group_scatter<F, MEM>(m, cache, lists, cnt, b, t, 32);
                    __syncwarp();
                }
            }
            if (tpr > 32) {
                if (lane == 0) ctl[4 + 2 * acc.par] = -1;
                acc.par ^= 1;
                named_bar(bar_id, tpr);
            }
        } else {
            for (;;) {
                named_bar(bar_id, tpr);
                const int cnt = ctl[4 + 2 * acc.par], own = ctl[5 + 2 * acc.par];
                acc.par ^= 1;
                if (cnt < 0) break;
                group_scatter<F, MEM>(m, cache, lists, cnt, own, t, tpr);
                named_bar(bar_id, tpr);
            }
        }
    }
}

// Sweeps [s0, s1) of replica r, whose state is built; `fresh`: sweep s0 is the
// run's first.
template <class F, class Z, int RULE, int MEM>
__device__ __forceinline__ void block_run(const SweepArgs& a, uint8_t* base, int bar_id, int t, int r, int s0, int s1,
                                          bool fresh, SweepAcc<F>& acc) {
    const int tpr = a.tpr;
    Z* zs = reinterpret_cast<Z*>(base + a.off_z);
    F* cache = reinterpret_cast<F*>(base + a.off_cache);
    int* ctl = reinterpret_cast<int*>(base + a.off_ctl);
    Commit* lists = reinterpret_cast<Commit*>(base + a.off_list);   // two lists of 32
    typename Num<F>::Acc* red = reinterpret_cast<typename Num<F>::Acc*>(base + a.off_red);
    uint8_t* stage = base + (a.off_blk >= 0 ? a.off_blk : 0);   // (not touched where blocks are not staged)
    const int nb = (a.m.n + 31) >> 5;
    BlockLane<F> q{};
    if (t < 32) {   // the first block, or all of one or two
        if (a.m.dense_rows && block_pair(tpr, nb)) {
            prepare_block<F, Z, RULE, MEM>(a, zs, stage, 0, s0, r, t, q);
        } else if (blocks_staged<MEM>(a)) {
            stage_block(a.m, stage, 0, t, true);
            if (nb == 2) stage_block(a.m, stage + kBlockStage, 1, t, true);
            stage_wait();
            __syncwarp();
        }
    }
    for (int s = s0; s < s1; ++s) {
        const bool flush = s + 1 == s1 || a.energy_trace != nullptr || a.best_states != nullptr ||
                           (Num<F>::is_float && a.refresh_interval > 0 && (s + 1) % a.refresh_interval == 0);
        block_sweep<F, Z, RULE, MEM>(a, zs, cache, ctl, lists, stage, bar_id, t, tpr, r, s, flush, acc, q);
        end_of_sweep<F, Z, KIND_QUIO, MEM, true>(a, zs, cache, red, t, tpr, bar_id, r, s, s == s0 && fresh, acc.e, acc.de,
                                      acc.drift);
    }
    stage_wait();   // no copy is in flight when the region is given up
}

}  // namespace dev
}  // namespace sa
