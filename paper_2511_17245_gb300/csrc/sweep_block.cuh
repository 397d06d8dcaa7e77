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
// lanes (the 32 x 32 couplings of the block, DevModel::blk_j), and the rest
// decide again.  The sequential order of Sect. 3.1 is kept exactly, changes are
// added to a field in that order, and nothing but warp shuffles separates two
// changes of a block.  Changes reach the other fields block by block.
//
// What bounds it: the chain of rounds, about 200 cycles each (decision, two
// ballots, one coupling row from L1).  Deciding level by level, or a window of
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
    int par;                         // blocked sweeps: which of the two commit lists is current
    int last;                        // and the block whose changes are not applied everywhere yet (-1: none)
};

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
    float pre[H];
    float sum = 0.f, comp = 0.f;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        pre[h] = 0.f;
        if (32 * h < n) {
            const uint32_t i0 = c0 + (uint32_t)(32 * h + lane);
            float w = 0.f;
            if (i0 <= c1) {
                if constexpr (Num<F>::is_float) w = ex2_ftz(fmaf(-vv.delta_ff(zf, v0f + (float)i0), b2, mb));
                else w = expf(-(Num<F>::to_f(vv.delta(z, lo + (long long)i0) - mn) * beta));
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

// ------------------------------------------------------------------ changes to the other fields
// Field j of a complete graph: the commits' couplings to it, in order.  Row k
// lists every j != k in order, so entry j - [j > k] of the row is J_kj.  Rows
// are read past L1 (each entry is used once) and eight at a time.
template <class F>
__device__ __forceinline__ F add_commits(const DevModel& m, F f, const Commit* list, int count, int j) {
    for (int c = 0; c < count; c += 8) {
        F w[8];
        int dz[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            dz[u] = 0;
            if (c + u < count) {
                const Commit e = list[c + u];
                dz[u] = e.y;
                w[u] = Coef<F>::adj_once(m, e.z + j - (j > e.x ? 1 : 0));
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (c + u < count) solo_add(&f, w[u], dz[u]);
    }
    return f;
}

// The commits' rows by columns, any graph: every thread of `nt` takes the next
// (commit, link) pair.  Columns of block `own` already have the change.
template <class F, int MEM>
__device__ __forceinline__ void scatter_commits(const DevModel& m, F* cache, const Commit* list, int count, int own,
                                                int t, int nt) {
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
            if (at[u] >= 0 && (col[u] >> 5) != own) {
                if constexpr (Num<F>::is_float) atomic_add_field<MEM>(cache + col[u], wt[u] * (float)dz[u]);
                else atomic_add_field<MEM>(cache + col[u], wt[u] * (long long)dz[u]);
            }
    }
}

// Rows with fewer links than this in all are scattered by the deciding warp.
constexpr int kScatterAlone = 96;

// The commits' rows by the `nt` threads t = 0..nt-1.  `ordered`: one commit
// after the other (bar_id < 0: the threads are one warp).
template <class F, int MEM>
__device__ __forceinline__ void group_scatter(const DevModel& m, F* cache, const Commit* list, int count, int own,
                                              bool ordered, int bar_id, int t, int nt) {
    if (!ordered) {
        scatter_commits<F, MEM>(m, cache, list, count, own, t, nt);
        return;
    }
    for (int c = 0; c < count; ++c) {
        const Commit e = list[c];
        for (int i = t; i < e.w; i += nt) {
            const int col = __ldg(m.adj_col + e.z + i);
            if ((col >> 5) != own) solo_add(cache + col, Coef<F>::adj(m, e.z + i), e.y);
        }
        if (c + 1 < count) {
            if (bar_id < 0) __syncwarp();
            else named_bar(bar_id, nt);
        }
    }
}

// ------------------------------------------------------------------ one block
// Decides block b (warp-collective) from the lanes' fields; on return f holds
// every change of the block, the list its commits.  Returns their number.
template <class F, class Z, int RULE>
__device__ __forceinline__ int decide_block(const SweepArgs& a, Z* zs, F& f, Commit* list, int b, int s, int r,
                                            float beta, float temp, float ratio, int lane, SweepAcc<F>& acc) {
    constexpr unsigned full = 0xffffffffu;
    const DevModel& m = a.m;
    const int kb = b * 32, k = kb + lane;
    const bool on = k < m.n;
    int4 x0 = make_int4(0, 0, 0, 0), x1 = x0;
    unsigned nbr = 0;   // earlier lanes of the block that share a term with this one
    if (on) {
        const int4* p = reinterpret_cast<const int4*>(m.idx_rec + k);
        x0 = __ldg(p);
        x1 = __ldg(p + 1);
        nbr = __ldg(m.blk_mask + k);
        // the block's coupling rows, one 128-byte line each (two for int64)
#pragma unroll
        for (int o = 0; o < (int)sizeof(F) / 4; ++o) prefetch_l1(Coef<F>::blk(m) + (size_t)k * 32 + 16 * o);
    }
    const int lo = x0.y;
    const uint32_t width = on ? (uint32_t)x0.z : 0u;
    F d;
    if constexpr (Num<F>::is_float) d = __uint_as_float((uint32_t)x1.z);
    else d = (long long)(((unsigned long long)(uint32_t)x1.w << 32) | (uint32_t)x1.z);
    const Words4 x = philox4x32_10((uint32_t)k, (uint32_t)s, (uint32_t)r, a.inst, a.key0, a.key1);
    const uint32_t zo = on ? (uint32_t)zs[k] : 0u;
    const long long z = (long long)lo + (long long)zo;
    const F* const blk = Coef<F>::blk(m) + (size_t)kb * 32 + lane;   // row p of the block: blk[32 p]
    long long v = z;
    int count = 0;
    auto trace = [&]() {
        if (a.trace != nullptr && r < a.trace_R && on)
            a.trace[((size_t)s * a.trace_R + r) * m.n + k] = (int32_t)v;
    };
    if constexpr (RULE == RULE_HEAT_BATH) {
        // one variable after the other, its range split over the lanes
        const int top = min(32, m.n - kb);
        for (int p = 0; p < top; ++p) {
            const uint32_t wp = __shfl_sync(full, width, p);
            if (wp == 0u) continue;
            VarView<F, KIND_QUIO> vv;
            vv.f = __shfl_sync(full, f, p);
            vv.d = __shfl_sync(full, d, p);
            const long long zp = __shfl_sync(full, z, p);
            const long long lp = __shfl_sync(full, lo, p);
            const uint32_t xp = __shfl_sync(full, x.x0, p);
            const bool fast = Num<F>::is_float && wp < 256u && lp > -(1 << 22) && lp + (long long)wp < (1 << 22);
            // the scalar or the warp-wide sum, whichever the level order takes
            // for this variable's level (the sums differ in their last bits)
            const bool wide = hb_warp_mode(__shfl_sync(full, x1.y, p), a.hb_tpr, m.max_width,
                                           Num<F>::is_float && m.max_width < 256u);
            long long vp;
            if (vv.linear()) {
                vp = heat_bath_linear(Num<F>::to_f(vv.lin_coef()), lp, wp, xp, beta);
            } else if (wide) {
                vp = heat_bath_warp<F, KIND_QUIO>(vv, zp, lp, wp, xp, beta, lane);
            } else {
                bool done = false;
                vp = zp;
                if constexpr (Num<F>::is_float) {
                    if (fast) {
                        vp = heat_bath_small_warp((float)vv.f, (float)vv.d, zp, lp, wp, xp, beta, temp, lane);
                        done = true;
                    }
                }
                if (!done) {
                    vp = wp < kChainValues ? heat_bath_chain<F>(vv, zp, lp, wp, xp, beta, lane)
                                  : heat_bath_general<F, KIND_QUIO>(vv, zp, lp, wp, xp, beta);
                }
            }
            if (lane == p) v = vp;
            if (vp != zp) {
                const F dp = vv.delta(zp, vp);
                const int dz = (int)(vp - zp);
                if constexpr (Num<F>::is_float) acc.de += lane == 0 ? (float)dp : 0.f;
                else acc.e += lane == 0 ? dp : 0;
                if (lane == p) {
                    list[count] = make_int4(k, dz, x0.w, x1.x);
                    zs[k] = (Z)(v - (long long)lo);
                    ++acc.changes;
                } else {
                    solo_add(&f, __ldg(blk + 32 * p), dz);
                }
                ++count;
            }
        }
        trace();
        return count;
    } else {
        long long prop = z;
        bool opt = false;
        if (width != 0u) {
            if (RULE == RULE_OPT) opt = unit_open_right(x.x2) < ratio;
            if (!opt) {
                const uint32_t j = pick_below(x.x0, width);
                prop = (long long)lo + (long long)(j >= zo ? j + 1u : j);
            }
        }
        unsigned open = __ballot_sync(full, width != 0u);   // lanes still to be decided
        while (open) {
            const bool mine = (open >> lane) & 1u;
            F de = F(0);
            bool chg = false;
            if (mine) {
                if (RULE == RULE_OPT && opt) {
                    VarView<F, KIND_QUIO> vv;
                    vv.f = f;
                    vv.d = d;
                    prop = opt_argmin<F, KIND_QUIO>(vv, z, lo, (long long)lo + (long long)width);
                }
                de = quio_delta<F>(f, d, z, prop);
                chg = prop != z && metropolis_accept<F>(de, x.x1, beta);
            }
            const unsigned c = __ballot_sync(full, chg);
            if (!c) break;
            // the first lane whose field one of the changes reaches decides again
            const unsigned late = __ballot_sync(full, mine && (nbr & c) != 0u);
            const int q = late ? __ffs(late) - 1 : 32;
            const unsigned done = late ? (1u << q) - 1u : full;
            unsigned com = c & done;
            if (chg && ((com >> lane) & 1u)) {
                v = prop;
                list[count + __popc(com & ((1u << lane) - 1u))] = make_int4(k, (int)(v - z), x0.w, x1.x);
                zs[k] = (Z)(v - (long long)lo);
                ++acc.changes;
                if constexpr (!Num<F>::is_float) acc.e += de;
            }
            count += __popc(com);
            const int dz = (int)(prop - z);
            while (com) {
                const int p = __ffs(com) - 1;
                com &= com - 1u;
                const F w = __ldg(blk + 32 * p);
                const int dp = __shfl_sync(full, dz, p);
                if (lane != p) solo_add(&f, w, dp);
                if constexpr (Num<F>::is_float) {   // summed in the visiting order, by one lane
                    const float ep = __shfl_sync(full, (float)de, p);
                    acc.de += lane == 0 ? ep : 0.f;
                }
            }
            open &= ~done;
        }
        trace();
        return count;
    }
}

// ------------------------------------------------------------------ one sweep
// Sweep s of replica r in blocks.  `flush`: the caller needs the state at the
// end of this sweep (a refresh, a trace, the outputs), so the last block's
// changes are applied before returning; otherwise they wait for the next sweep.
//
// Complete graphs: while warp 0 decides block b, the other warps add the changes
// of block b - 1 to every field outside of blocks b - 1 and b (each field by one
// thread, its rows eight loads deep); warp 0 adds them to block b's fields
// itself when it starts on them.  One barrier per block.
// Other graphs: warp 0 decides, then the group scatters the block's rows by
// their columns; short rows are scattered by warp 0 without waking the others.
// Float models whose every level holds one variable keep the order of the
// additions (one commit at a time).
template <class F, class Z, int RULE, int MEM>
__device__ __forceinline__ void block_sweep(const SweepArgs& a, Z* zs, F* cache, int* ctl, Commit* lists, int bar_id,
                                            int t, int tpr, int r, int s, bool flush, SweepAcc<F>& acc) {
    const DevModel& m = a.m;
    const int lane = t & 31;
    const float beta = __ldg(a.beta + s);
    const float temp = 1.f / beta;
    const float ratio = __ldg(a.ratio + s);
    const int nb = (m.n + 31) >> 5;
    if (m.dense_rows) {
        for (int b = 0; b < nb; ++b) {
            const Commit* prev = lists + 32 * (acc.par ^ 1);
            const int np = acc.last >= 0 ? ctl[acc.par ^ 1] : 0;
            if (t < 32) {
                const int k = b * 32 + lane;
                F f = F(0);
                if (k < m.n) {
                    f = cache[k];
                    if (acc.last != b) f = add_commits<F>(m, f, prev, np, k);
                }
                const int cnt = decide_block<F, Z, RULE>(a, zs, f, lists + 32 * acc.par, b, s, r, beta, temp, ratio,
                                                         lane, acc);
                if (k < m.n) cache[k] = f;
                if (lane == 0) ctl[acc.par] = cnt;
            }
            if (np > 0 && (t >= 32 || tpr == 32)) {
                const int nt = tpr > 32 ? tpr - 32 : 32;
                for (int j = tpr > 32 ? t - 32 : t; j < m.n; j += nt) {
                    const int bj = j >> 5;
                    if (bj != b && bj != acc.last) cache[j] = add_commits<F>(m, cache[j], prev, np, j);
                }
            }
            named_bar(bar_id, tpr);
            acc.par ^= 1;
            acc.last = b;
        }
        if (flush) {
            const int np = ctl[acc.par ^ 1];
            for (int j = t; j < m.n; j += tpr)
                if ((j >> 5) != acc.last) cache[j] = add_commits<F>(m, cache[j], lists + 32 * (acc.par ^ 1), np, j);
            named_bar(bar_id, tpr);
            acc.last = -1;
        }
    } else {
        // commands to the other warps: {commits or -1, their block}, in two
        // alternating places, so that one is read before it is written again
        const bool ordered = Num<F>::is_float && m.n_levels == m.n;
        if (t < 32) {
            for (int b = 0; b < nb; ++b) {
                const int k = b * 32 + lane;
                F f = k < m.n ? cache[k] : F(0);
                const int cnt = decide_block<F, Z, RULE>(a, zs, f, lists, b, s, r, beta, temp, ratio, lane, acc);
                if (k < m.n) cache[k] = f;
                __syncwarp();
                if (cnt == 0 || nb == 1) continue;
                const int links = __reduce_add_sync(0xffffffffu, lane < cnt ? lists[lane].w : 0);
                if (tpr > 32 && links > kScatterAlone) {
                    if (lane == 0) {
                        ctl[4 + 2 * acc.par] = cnt;
                        ctl[5 + 2 * acc.par] = b;
                    }
                    acc.par ^= 1;
                    named_bar(bar_id, tpr);
                    group_scatter<F, MEM>(m, cache, lists, cnt, b, ordered, bar_id, t, tpr);
                    named_bar(bar_id, tpr);
                } else {
                    group_scatter<F, MEM>(m, cache, lists, cnt, b, ordered, -1, t, 32);
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
                group_scatter<F, MEM>(m, cache, lists, cnt, own, ordered, bar_id, t, tpr);
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
    for (int s = s0; s < s1; ++s) {
        const bool flush = s + 1 == s1 || a.energy_trace != nullptr || a.best_states != nullptr ||
                           (Num<F>::is_float && a.refresh_interval > 0 && (s + 1) % a.refresh_interval == 0);
        block_sweep<F, Z, RULE, MEM>(a, zs, cache, ctl, lists, bar_id, t, tpr, r, s, flush, acc);
        end_of_sweep<F, Z, KIND_QUIO>(a, zs, cache, red, t, tpr, bar_id, r, s, s == s0 && fresh, acc.e, acc.de,
                                      acc.drift);
    }
}

}  // namespace dev
}  // namespace sa
