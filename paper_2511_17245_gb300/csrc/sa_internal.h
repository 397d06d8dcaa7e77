// sa_internal.h -- device model layout and kernel arguments shared by the
// host-side model compiler and launchers (api.cu, batch.cu, noalloc.cu,
// server.cu) and the CUDA kernels.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

namespace sa {

enum Kind : int32_t { KIND_QUIO = 0, KIND_HUIO = 1 };

// Per-variable metadata, 16 bytes, read once per attempt.
struct VarMeta {
    int32_t lo;           // l_k
    uint32_t width;       // u_k - l_k (0 = fixed variable)
    int32_t link_begin;   // QUIO: first adjacency entry; HUIO: first incidence entry
    int32_t link_len;     // number of adjacency / incidence entries
};

// Per-variable record in dependency-level order, 32 bytes, everything one
// attempt needs besides the replica state.  aux holds J_kk (QUIO; fp32 bits or
// int64) or the exponent mask Omega_k (HUIO).
struct alignas(16) LevelRec {
    int32_t k;
    int32_t lo;
    uint32_t width;
    int32_t link_begin;
    int32_t link_len;
    int32_t slot_base;
    uint32_t aux0, aux1;
};

// Device-resident compiled model.  All pointers are device pointers into one
// allocation.  For integer models the *_i arrays are used; for float models
// the *_f arrays drive the sweep and the *_d arrays the FP64 refresh.
struct DevModel {
    int32_t n;
    int32_t kind;
    int32_t is_float;
    int32_t n_levels;
    uint32_t max_width;         // largest u_k - l_k
    int32_t dense_rows;         // QUIO on a complete graph: row k lists every j != k in increasing order
    const VarMeta* meta;        // [n]
    const int32_t* lvl_ptr;     // [n_levels + 1]
    const int32_t* lvl_vars;    // [n]: variables grouped by dependency level
    const LevelRec* lvl_rec;    // [n]: their records, same order
    // models with narrow levels (plan_block_model), swept in blocks of 32
    // consecutive variables; null otherwise
    const LevelRec* idx_rec;    // [n]: records in index order, slot_base = width of the variable's level
    const uint32_t* blk_mask;   // [n]: bit j set iff variable 32 (k / 32) + j < k shares a term with k
    const int32_t* blk_w;       // [32 ceil(n / 32)][32]: J_kj of the variables j of k's block (fp32 bits or int32)
    const int32_t* blk_part;    // fp32 models [n][kRowParts]: first entry of row k, from the row's start, whose
                                // column is in part p of the columns or a later one (plan_row_part)
    const int64_t* blk_i;       // the same in int64, when some J_kj does not fit int32 (blk_w is not read then)

    // QUIO (every term of total degree <= 2):
    //   E = c + sum_k lin_k z_k + sum_k diag_k z_k^2 + sum_{i<j} J_ij z_i z_j
    // [n]: {k, first entry of row k with a column above k, end of row k, 0}, by
    // the number of those entries (descending) and the first one's place in its
    // group of four, so that a warp's lanes walk alike
    const int32_t* up_rec;
    // normal fp32 couplings of sparse models with small values (plan_pair_list): every
    // pair once, {smaller variable | larger << 16, fp32 bits of J}, by rows; null otherwise
    const int32_t* up_pair;
    int32_t n_pairs;
    int32_t z_base;             // smallest lower bound
    uint32_t z_span;            // largest upper bound minus z_base
    const int32_t* adj_col;     // symmetric adjacency, both directions
    const int64_t* adj_i;
    const float* adj_f;
    const double* adj_d;        // null when the coefficients were given as fp32
    const int64_t* lin_i;
    const float* lin_f;
    const double* lin_d;
    const int64_t* diag_i;
    const float* diag_f;
    const double* diag_d;

    // HUIO: per-variable coefficient slots a_k^(m), m in Omega_k
    int32_t n_slots;
    int32_t n_iterms;           // interaction terms (two or more distinct variables)
    const int32_t* slot_base;   // [n]
    const uint64_t* omega;      // [n]: bit m set iff z_k^m appears in some term
    const int64_t* aconst_i;    // [n_slots]: single-variable terms J_{k..k} (constant part)
    const float* aconst_f;
    const double* aconst_d;
    const int32_t* inc_term;    // incidence of variable s: interaction terms containing s
    const int32_t* inc_exp;     //   and the exponent of s in that term
    // per incidence, 16 int32 (four 16-byte groups): {coefficient (int64, or
    // fp32 bits and 0), exponent of s | number of other members (0..3) << 8 |
    // 1 << 16 when every exponent is 1 (or -1 for terms of more than 4
    // members), the other members' exponents packed e1 | e2 << 8 | e3 << 16},
    // {their variables v1..v3, term}, {their coefficient slots (slot_base[v] +
    // index of the exponent), 0}, {their lower bounds, 0}; null where inc16 is not
    const int32_t* inc_rec;
    // multilinear models of at most 65,534 variables, few of them in no term, with
    // one lower bound, terms of at most 4 members and coefficients that fit 32
    // bits: the same in one 16-byte group, {coefficient (int32 or fp32 bits), v1 | v2 << 16, v3, 0} with
    // 0xFFFF for no variable (variable v's slot is v); null otherwise
    const int32_t* inc16;
    const int32_t* term_ptr;    // [n_iterms + 1] into mem_var / mem_exp
    const int32_t* mem_var;     // members (distinct variables) of interaction terms
    const int32_t* mem_exp;     // their exponents
    const int64_t* tcoef_i;     // [n_iterms]
    const float* tcoef_f;
    const double* tcoef_d;

    int64_t const_i;            // empty multiset
    double const_d;
};

enum Rule : int32_t { RULE_METROPOLIS = 0, RULE_HEAT_BATH = 1, RULE_OPT = 2 };

// Arguments of the sweep kernel (passed by value).
struct SweepArgs {
    DevModel m;
    int32_t R;                  // replicas
    int32_t S;                  // sweeps
    uint32_t key0, key1;        // Philox key
    uint32_t inst;              // fourth counter word
    int32_t refresh_interval;   // float models
    const float* beta;          // [S]
    const float* ratio;         // [S]
    const int32_t* init_states; // [R][n] or null
    int32_t* out_states;        // [R][n]
    void* out_energies;         // int64 or double [R]
    unsigned long long* out_accepts;  // [R] or null
    int32_t* trace;             // [S][trace_R][n] or null
    int32_t trace_R;
    void* energy_trace;         // [S][R] or null
    unsigned int* drift_bits;   // max refresh drift (float bits, atomicMax) or null
    uint8_t* gstate;            // per-replica state slabs when not on chip
    int64_t rep_bytes;          // bytes of one replica's state region
    int32_t off_z, off_cache, off_ctl, off_list, off_red;
    int32_t off_blk;            // blocked sweeps: two staged blocks (kBlockStage bytes each; -1: not staged)
    int32_t off_lvl;            // level boundaries staged in the replica region (-1: read from the model)
    int32_t blocked;            // sweep in blocks of 32 variables (the model has idx_rec)
    int32_t hb_tpr;             // threads per replica that decide the form of heat-bath sums (hb_warp_mode)
    int32_t _pad0;
    int32_t rpc;                // replicas per block
    int32_t tpr;                // threads per replica (multiple of 32)
    int32_t heavy_links;        // link_len above which updates are cooperative
    int32_t list_cap;           // capacity of the cooperative update list
    // time-sliced runs (sweep_sliced_kernel): per-replica regions through which
    // a replica's state passes from one chunk of sweeps to the next, the number
    // of finished chunks per replica, the task counter and an error word
    uint8_t* handoff;
    unsigned int* handoff_flag; // [R]: chunks of the replica finished (and saved)
    int64_t handoff_bytes;      // bytes of one region: off_ctl + 24 per thread, rounded to 16
    unsigned int* status;       // [0] bit 0: a handoff wait gave up (that replica's outputs are not
                                // written); [1]: task counter
    int32_t* best_states;       // [R][N] or null: lowest-energy state at a sweep end
    void* best_energies;        // [R] (int64 or double): its tracked energy
};

// One unit of batched work: one replica of one instance.
struct BatchUnit {
    int32_t inst;
    int32_t replica;
};

// Arguments of the persistent batched kernel.
struct BatchArgs {
    const SweepArgs* insts;     // per-instance arguments (device table)
    const BatchUnit* units;     // ordered by decreasing cost
    int32_t n_units;
    unsigned int* counter;      // next unit (reset to 0 before every launch)
    int64_t slot_bytes;         // state region of one thread group (max over instances)
    int32_t rpc, tpr;
    uint8_t* gstate;            // per-group regions when the state is not on chip
};

// ------------------------------------------------------------------ serving
// One admitted request of the server: the kernel arguments of its run (the
// fields of SweepArgs, with the layout for the serving kernel's group size)
// and which compiled variant runs it.  Written by the host into host-mapped
// memory before the request's units are published.
struct ServeReq {
    SweepArgs args;
    int32_t variant;            // serve_variant(...)
    int32_t n_units;            // replicas
};

// A unit of serving work: one replica of one admitted request.
struct ServeUnit {
    int32_t req;                // request slot
    int32_t replica;
};

// Host-mapped control words of the serving queue.
struct ServeCtl {
    volatile uint32_t tail;     // units published so far (host writes)
    volatile uint32_t stop;     // nonzero: groups leave once the queue is empty
};

// Arguments of the persistent serving kernel.
struct ServeArgs {
    const ServeReq* reqs;       // [max_reqs], host-mapped
    const ServeUnit* units;     // ring of `cap` units, host-mapped
    const ServeCtl* ctl;        // host-mapped
    unsigned int* head;         // device: next unit to claim
    unsigned int* req_units_done;   // device: [max_reqs] finished units per request slot
    unsigned int* req_done;     // host-mapped: [max_reqs] set to 1 when a request's last unit finished
    uint32_t cap;               // ring capacity (a power of two)
    int32_t tpr, rpc;
    int32_t _pad0;
    int64_t slot_bytes;         // shared-memory state region of one thread group
    uint32_t idle_polls;        // empty-queue polls (about 2 us each) before a group leaves
    uint32_t _pad1;
};

// Variant index of a request for the serving kernel: rule, model kind,
// coefficient class and 2- or 4-byte state offsets.
inline int serve_variant(int rule, int kind, int is_float, int zbytes) {
    return rule + 3 * (kind + 2 * (is_float + 2 * (zbytes > 2 ? 1 : 0)));
}

// Arguments of the energy kernel.
struct EnergyArgs {
    DevModel m;
    const int32_t* states;      // [n_states][n]
    int64_t n_states;
    void* energies;             // int64 or double
    int32_t* bad;               // set to 1 if a value lies outside its bounds
};

// Read-only view of a compiled model for translation units other than api.cu.
struct ModelView {
    DevModel dm;
    int device;
    int32_t n;
    int is_float;
    int max_exp;
    int zbytes;
    int64_t cache_elems;
    int32_t n_levels;
    int32_t max_link_len;       // longest neighbour / incidence list
    int64_t n_links;
    double de_max, de_min;
};

// Threads per replica for a launch whose caller left the choice to the library.
// `tpr` is the choice from the level widths; when the block's replicas leave
// thread slots unused (few replicas per SM) and some variable's update list is
// longer than `heavy_links` (the lists the whole group updates together), the
// spare slots go to the replicas.  Integer results do not depend on the shape.
inline int grow_threads_per_replica(int tpr, int32_t max_link_len, int heavy_links, int replicas,
                                    int replicas_per_block, int sms) {
    if (max_link_len <= heavy_links) return tpr;
    int per_block = replicas_per_block > 0 ? replicas_per_block : (replicas + sms - 1) / (sms > 0 ? sms : 1);
    per_block = per_block < 1 ? 1 : (per_block > 15 ? 15 : per_block);
    int grown = (512 / per_block) / 32 * 32;
    if (grown > 256) grown = 256;
    return grown > tpr ? grown : tpr;
}

// ------------------------------------------------------------------ run planning
// Host-side planning shared by every entry point that launches the sweep
// kernel (sa_run, sa_run_noalloc, batches).  Pure arithmetic: no CUDA calls,
// so that the same rules can be checked on a machine without a GPU.

// What the planner needs to know about a compiled model.
struct PlanModel {
    int32_t n;
    int32_t n_levels;
    int32_t kind;               // KIND_QUIO / KIND_HUIO
    int32_t is_float;
    int32_t zbytes;             // bytes of one state offset z_k - l_k
    int32_t max_link_len;
    int64_t cache_elems;        // QUIO: n fields; HUIO: coefficient slots
    int32_t block_model;        // the model holds the tables of the blocked sweep
    int32_t dense_rows;         // complete graph
    int32_t mean_links;         // mean length of the neighbour lists
    uint32_t max_width;         // largest u_k - l_k
};

inline PlanModel plan_model(const ModelView& v) {
    return PlanModel{v.n, v.n_levels, v.dm.kind, v.is_float, v.zbytes, v.max_link_len, v.cache_elems,
                     v.dm.idx_rec != nullptr, v.dm.dense_rows, (int32_t)(v.n_links / (v.n > 0 ? v.n : 1)),
                     v.dm.max_width};
}

// ------------------------------------------------------------------ blocked sweeps
// A level costs a group barrier, a Philox block and an L2 round trip whatever
// its width; a block of 32 variables costs one of each plus a short round per
// colliding change.  kBlockWidth is the mean level width up to which models hold
// the tables of the blocked sweep (QUIO) and the Metropolis rules use it: 64 /
// 1024 replicas x 20 sweeps, blocks against the level order, int64, 320 variables
// of width 7 0.67 / 1.02 against 1.96 / 2.15 ms, 1000 of width 15 2.1 / 3.4 against
// 5.6 / 5.8; fp32, 1000 of width 13 2.25 / 3.16 against 4.5 / 4.8.
constexpr int kBlockWidth = 16;

// The heat bath's limit, by the number of values of the widest range.  A block
// decides wide ranges one variable after the other by one warp, a level side by
// side by all of them, so the limit falls as a decision grows.  Times in ms of 5
// sweeps, 64 / 1024 replicas, blocks against levels (1000 variables, * 200):
//   fp32    64 values: width 2.3   5.6 / 11.5 against 6.2 / 14.1; * 2.7  1.08 / 1.44 against 0.95 / 1.32
//          128 values: width 2.3   6.9 / 13.0 against 6.4 / 14.6; * 2.7  1.29 / 1.64 against 1.03 / 1.40
//          256 values: width 1.7  11.2 / 20.0 against 10.5 / 22.5;  2.3  10.8 / 15.8 against 7.8 / 16.2
//         1024 values: width 1.3  15.3 / 29.1 against 16.3 / 33.2;  1.7  14.6 / 25.4 against 12.6 / 26.3
//   int64   48 values: * 2.7  2.4 / 3.1 against 3.0 / 3.9 (wide levels begin at 57)
//          256 values: width 1.4  13.3 / 28.4 against 13.7 / 27.3;  1.8  12.7 / 23.9 against 10.9 / 21.9
//         1024 values: width 1.1  21.2 / 42.4 against 23.8 / 44.1; * 1.2  4.1 / 5.8 against 4.3 / 5.8
inline double block_width_heat(bool is_float, uint32_t max_width) {
    const int64_t values = (int64_t)max_width + 1;
    if (is_float) return values <= 128 ? 2.5 : (values <= 256 ? 1.75 : 1.5);
    return values <= 56 ? 3.0 : (values <= 256 ? 1.5 : 1.1);
}

inline bool plan_block_model(int32_t n, int32_t n_levels) { return (int64_t)n <= (int64_t)kBlockWidth * n_levels; }

// Whether a run of this model sweeps in blocks (`allowed`: the caller did not
// ask for the level order).
inline bool plan_blocked(const PlanModel& m, int rule, bool allowed) {
    if (!m.block_model || !allowed) return false;
    return rule != RULE_HEAT_BATH || (double)m.n <= block_width_heat(m.is_float != 0, m.max_width) * (double)m.n_levels;
}

// Whether the model holds the pair list that the energies of states are summed
// from: variables in 16 bits, values whose product two of them have exactly in
// fp32, and short rows (rows of 64 entries and more fill a thread's groups of
// four without it, and the list of a complete graph would be half its adjacency).
inline bool plan_pair_list(int32_t n, int64_t lo, int64_t hi, int64_t pairs) {
    return n <= 65536 && lo > -4096 && hi < 4096 && pairs <= 32 * (int64_t)n;
}

// Parts of the columns (whole blocks of 32) that the warps of a group take when
// they add a block's changes to fp32 fields in order; columns of one part.
constexpr int kRowParts = 16;
inline int32_t plan_row_part(int32_t n) { return ((n + 31) / 32 + kRowParts - 1) / kRowParts * 32; }

// Bytes of one block staged on chip: couplings (32 x 32 x 4), records, masks.
constexpr int kBlockStage = 4096 + 32 * (int)sizeof(LevelRec) + 128;

// Threads that a replica of a blocked sweep can use: one warp decides; the
// others add its changes to the other fields (complete graphs: every field,
// several rows deep; else the rows' links).
inline int plan_blocked_threads(const PlanModel& m) {
    if (m.n <= 32) return 32;
    // complete fp32 graphs, 152 replicas x 20 sweeps, ms with 64 / 128 / 192 / 256 /
    // 384 / 512 threads:
    //    200 variables  0.70   0.62   0.68   0.71   0.72   0.73
    //    500            3.33   1.76   1.62   1.73   2.13   2.55
    //   1000           12.8    6.58   4.87   3.97   4.17   5.00
    //   1998           50.6   25.9   16.3   13.2   14.1   11.4
    // (600 replicas, four to a block of at most 512 threads: 1000 variables 11.7 ms
    // with the 128 that fit, 13.7 with 192 and 16.5 with 384)
    if (m.dense_rows) {
        const int want = (m.n * 3 / 8 + 31) / 32 * 32;
        return want > 512 ? 512 : (want < 128 && m.n > 64 ? 128 : want);
    }
    const int work = 4 * m.mean_links < m.n ? 4 * m.mean_links : m.n;
    const int want = 32 + (work + 31) / 32 * 32;
    return want > 512 ? 512 : want;
}

// Threads that a replica of a level-by-level sweep can use: twice the mean level
// width, so that nearly every level is one round (levels of a random graph are
// up to twice as wide as the mean).  1501 variables of mean degree 16, 36 levels,
// 512 replicas x 100 sweeps: 32 threads 13.9 ms, 64 9.4, 96 9.0, 128 9.6.
inline int plan_level_threads(const PlanModel& m, int tpr) {
    const int levels = m.n_levels > 0 ? m.n_levels : 1;
    int want = (2 * (m.n / levels) + 31) / 32 * 32;
    want = want > 256 ? 256 : want;
    return want > tpr ? want : tpr;
}

// Per-replica state layout and launch shape of one run.
struct RunPlan {
    int32_t tpr;                // threads per replica (whole warps)
    int32_t rpc;                // replicas per block
    int32_t blocks;
    int32_t heavy_links;        // update lists above this length go to the cooperative list
    int32_t list_cap;           // entries of the cooperative list (list_words each)
    int32_t in_global;          // replica state in global memory instead of shared memory
    int64_t rep_bytes;          // bytes of one replica's state region
    int64_t shared_bytes;       // dynamic shared memory of one block
    int32_t off_z, off_cache, off_ctl, off_list, off_red, off_lvl, off_blk;
    int32_t blocked, hb_tpr;    // see SweepArgs (set by plan_run)
};

inline int64_t plan_round16(int64_t x) { return (x + 15) / 16 * 16; }

// Words of an entry of the cooperative list (five are used; QUIO's lists hold a
// blocked sweep's two lists of 32 16-byte commits as well).
constexpr int list_words(int kind) { return kind == KIND_HUIO ? 5 : 6; }
// Bytes that the shorter entries save in the region of a HUIO replica, for slots
// of unused variables (see compile_terms).
constexpr int64_t kSlotSlack = 256 * 4;

// State layout of one replica for `tpr` threads: offsets z_k - l_k (zbytes
// each), the cache (int64 or fp32), the control words (three list counters or
// the commit counts and commands of a blocked sweep), the cooperative update
// list or a blocked sweep's two commit lists, the reduction scratch (one 8-byte word
// per warp) and, when it takes at most 16 KB, the level boundary table.  (The
// staged blocks of a blocked sweep come after it where they fit, see plan_run.)
// `zbytes` may exceed the model's own (a batch uses its widest).  QUIO rows are
// cheap per entry (one atomic) and go inline up to 64 links; HUIO incidences
// cost a term product each, and every list of them goes to the group.
inline int64_t plan_layout(const PlanModel& m, int zbytes, int tpr, RunPlan* p) {
    const bool huio = m.kind == KIND_HUIO;
    const int64_t fsize = m.is_float ? 4 : 8;
    p->tpr = tpr;
    p->heavy_links = huio ? 0 : 64;
    p->list_cap = huio ? 256 : 64;
    p->off_z = 0;
    p->off_cache = (int32_t)plan_round16((int64_t)m.n * zbytes);
    p->off_ctl = (int32_t)plan_round16(p->off_cache + m.cache_elems * fsize);
    p->off_list = p->off_ctl + 112;
    p->off_red = (int32_t)plan_round16(p->off_list + (int64_t)p->list_cap * list_words(m.kind) * 4);
    const int64_t lvl_bytes = (int64_t)(m.n_levels + 1) * 4;
    const int64_t off_lvl = plan_round16(p->off_red + (int64_t)(tpr / 32) * 8);
    const bool lvl_on_chip = lvl_bytes <= 16384;
    p->off_lvl = lvl_on_chip ? (int32_t)off_lvl : -1;
    p->off_blk = -1;
    p->rep_bytes = plan_round16(off_lvl + (lvl_on_chip ? lvl_bytes : 0));
    return p->rep_bytes;
}

// Launch shape of a single-model run of R replicas.  tpr_req / rpc_req <= 0
// leave the choice to the library: tpr from the mean level width (half of it,
// rounded up to whole warps, 32..256), grown by grow_threads_per_replica for
// long update lists; rpc as many replicas as shared memory and 512 threads
// allow, but no more than needed to spread the replicas over the SMs.  Returns
// nullptr, or a message describing the invalid request.
inline const char* plan_run_shape(const PlanModel& m, int32_t R, int32_t tpr_req, int32_t rpc_req, bool force_global,
                                  int sms, int64_t smem_max, RunPlan* p) {
    int tpr = tpr_req;
    if (tpr <= 0) {
        const double mean_w = (double)m.n / (double)(m.n_levels > 0 ? m.n_levels : 1);
        int want = (int)(mean_w / 2.0);
        if ((double)want < mean_w / 2.0) ++want;
        tpr = (want + 31) / 32 * 32;
        tpr = tpr < 32 ? 32 : (tpr > 256 ? 256 : tpr);
    }
    if (tpr % 32 != 0 || tpr > 512 || tpr < 32) return "threads_per_replica must be a multiple of 32, <= 512";
    if (tpr_req <= 0)
        tpr = grow_threads_per_replica(tpr, m.max_link_len, m.kind == KIND_HUIO ? 8 : 64, R, rpc_req, sms);
    const int64_t rep = plan_layout(m, m.zbytes, tpr, p);
    int fit = (int)(smem_max / rep);
    const int cap = 15 < 512 / tpr ? 15 : 512 / tpr;
    fit = fit < cap ? fit : cap;
    const bool in_global = fit < 1 || force_global;
    int rpc = rpc_req;
    if (rpc <= 0) {
        int target = (R + (sms > 0 ? sms : 1) - 1) / (sms > 0 ? sms : 1);
        target = target < 1 ? 1 : target;
        rpc = in_global ? (target < cap ? target : cap) : (fit < target ? fit : target);
    }
    if (rpc < 1 || rpc > 15 || rpc * tpr > 512) return "replicas_per_block out of range";
    if (!in_global && rpc > fit) return "replicas_per_block exceeds shared memory";
    p->rpc = rpc;
    p->in_global = in_global ? 1 : 0;
    p->blocks = (R + rpc - 1) / rpc;
    p->shared_bytes = in_global ? 0 : (int64_t)rpc * rep;
    return nullptr;
}

// Plan of a single-model run: plan_run_shape, and for blocked sweeps whose
// caller left the thread count open, the threads that such a sweep can use
// within 512 per block.
inline const char* plan_run(const PlanModel& m, int rule, bool allow_blocks, int32_t R, int32_t tpr_req,
                            int32_t rpc_req, bool force_global, int sms, int64_t smem_max, RunPlan* p) {
    if (const char* err = plan_run_shape(m, R, tpr_req, rpc_req, force_global, sms, smem_max, p)) return err;
    const int32_t hb_tpr = p->tpr;
    // (the shape does not depend on allow_blocks, so that float energies, summed
    // in FP64 over the replica's threads, are the same bits either way)
    const bool blocked = plan_blocked(m, rule, true);
    if (tpr_req <= 0) {
        const int rpc = p->rpc;
        int tpr = blocked ? plan_blocked_threads(m) : plan_level_threads(m, p->tpr);
        const int cap = 512 / rpc / 32 * 32;
        tpr = tpr > cap ? cap : tpr;
        RunPlan q{};
        // more threads per replica grow its region a little: keep the first plan if that no longer fits
        if (plan_run_shape(m, R, tpr, rpc, force_global, sms, smem_max, &q) == nullptr && q.in_global == p->in_global)
            *p = q;
    }
    p->blocked = blocked && allow_blocks ? 1 : 0;
    p->hb_tpr = hb_tpr;
    // staged blocks only where there is room: they never change which shapes and
    // placements are possible
    if (p->blocked && !p->in_global && (p->rep_bytes + 2 * kBlockStage) * p->rpc + 1024 <= smem_max) {
        p->off_blk = (int32_t)p->rep_bytes;
        p->rep_bytes += 2 * kBlockStage;
        p->shared_bytes = p->rep_bytes * p->rpc;
    }
    return nullptr;
}

// ------------------------------------------------------------------ batch launch shape
// One thread group's place in a batch kernel besides its replica's state: the
// arguments of its present instance and the unit it claimed.  They lie in the
// dynamic shared memory behind the state regions, one per group of the launch, so
// that what the shape counts is what the kernel uses.
struct alignas(16) BatchGroup {
    SweepArgs args;
    int32_t unit;
};

struct BatchShape {
    int32_t rpc, per_sm;        // replicas per block, blocks per SM of the persistent grid
    int32_t in_global;          // replica state in global slabs
    int32_t staged;             // blocked instances stage their blocks behind the region
    int64_t slot_bytes;         // bytes of one replica's region
    int64_t shared_bytes;       // dynamic shared memory of one block
};

// Shape of a batch launch whose largest replica region takes `slot` bytes at
// `tpr` threads per replica.  rpc_req <= 0: as many replicas per block as shared
// memory and 512 threads allow.
inline const char* plan_batch_shape(int64_t slot, int tpr, int rpc_req, bool any_blocked, int64_t smem_max,
                                    BatchShape* p) {
    constexpr int64_t group = (int64_t)sizeof(BatchGroup);
    const int cap = 15 < 512 / tpr ? 15 : 512 / tpr;
    const int64_t room = smem_max / (slot + group);
    const int fit = room < cap ? (int)room : cap;
    p->in_global = fit < 1 ? 1 : 0;
    p->rpc = rpc_req > 0 ? rpc_req : (p->in_global ? cap : fit);
    if (p->rpc < 1 || p->rpc > 15 || p->rpc * tpr > 512) return "batch launch shape out of range";
    if (!p->in_global && p->rpc > fit) return "replicas_per_block exceeds shared memory";
    // persistent grid: as many blocks as fit on the GPU at once (1 per SM with
    // large shared use; 1 KB of each block is the system's), registers for up to
    // 128 per thread
    auto shared = [&](int64_t s) { return (p->in_global ? 0 : p->rpc * s) + p->rpc * group; };
    auto fits = [&](int64_t s) { return (int)((smem_max + 1024) / (shared(s) + 1024)); };
    int per_sm = 2048 / (p->rpc * tpr);
    if (per_sm > 65536 / (p->rpc * tpr * 128)) per_sm = 65536 / (p->rpc * tpr * 128);
    if (per_sm > fits(slot)) per_sm = fits(slot);
    p->per_sm = per_sm < 1 ? 1 : per_sm;
    // blocked instances stage their blocks where there is room
    p->staged = any_blocked && !p->in_global && shared(slot + 2 * kBlockStage) <= smem_max &&
                fits(slot + 2 * kBlockStage) >= p->per_sm;
    p->slot_bytes = slot + (p->staged ? 2 * kBlockStage : 0);
    p->shared_bytes = shared(p->slot_bytes);
    return nullptr;
}

// ------------------------------------------------------------------ time-sliced runs
// When R replicas exceed the P thread groups that can be resident at once, a
// plain launch runs ceil(R / P) waves and the last one leaves slots idle.  A
// time-sliced launch instead cuts every replica's S sweeps into C chunks of K
// sweeps and lets the resident groups claim (replica, chunk) tasks from one
// counter in chunk-major order: task q is chunk q / R of replica q % R.  A
// chunk after the first waits for its replica's previous chunk, restores the
// state that chunk saved and saves its own for the next.  Every task's
// predecessor was claimed earlier by a resident group, so the chain of waits
// always ends at a running task; and with R >= P a predecessor was claimed
// about R tasks earlier, so it has usually finished.  Claiming tasks one by one
// balances the groups by the actual cost of the sweeps (which varies along the
// schedule), the last round of tasks being one chunk long.
constexpr int kSliceChunks = 16;

// Sweeps per chunk of a time-sliced run of S sweeps (at most kSliceChunks chunks).
inline
#ifdef __CUDACC__
__host__ __device__
#endif
int32_t slice_chunk_sweeps(int32_t S) {
    return (S + kSliceChunks - 1) / kSliceChunks;
}

// Per-sweep table read by the kernel: tab[s] = fp32(1 / T_s) with the geometric
// schedule T_s = T_max (T_min / T_max)^(s / (S - 1)) of Sect. 3.1 (T_0 = T_max
// when S = 1) or the caller's temperatures, and tab[S + s] = the OTM ratio
// r_s = fp32(s) / fp32(S - 1) of Sect. 3.3.3 (0 when S = 1).  t_max and t_min
// both <= 0 select the Sect. 3.4 temperatures -dE_max / ln(1/2) and
// -dE_min / ln(0.001).  Returns nullptr or an error message.
inline const char* plan_schedule(double de_max, double de_min, int32_t S, double t_max, double t_min,
                                 const double* temps, float* tab) {
    if (!temps) {
        if (t_max <= 0 && t_min <= 0) {
            t_max = -de_max / std::log(0.5);
            t_min = -de_min / std::log(0.001);
        } else if (!(t_max > 0 && t_min > 0) || !std::isfinite(t_max) || !std::isfinite(t_min)) {
            return "t_max and t_min must both be positive (or both <= 0 for defaults)";
        }
    }
    for (int32_t s = 0; s < S; ++s) {
        double T;
        if (temps) {
            T = temps[s];
            if (!(T > 0) || !std::isfinite(T)) return "temperatures must be positive";
        } else {
            const double frac = S > 1 ? (double)s / (double)(S - 1) : 0.0;
            T = t_max * std::pow(t_min / t_max, frac);
        }
        tab[s] = (float)(1.0 / T);
        tab[S + s] = S > 1 ? (float)s / (float)(S - 1) : 0.0f;
    }
    return nullptr;
}

// Copies the layout and shape of a plan into the kernel arguments.
inline void plan_apply(const RunPlan& p, SweepArgs& a) {
    a.rep_bytes = p.rep_bytes;
    a.off_z = p.off_z;
    a.off_cache = p.off_cache;
    a.off_ctl = p.off_ctl;
    a.off_list = p.off_list;
    a.off_red = p.off_red;
    a.off_lvl = p.off_lvl;
    a.off_blk = p.off_blk;
    a.rpc = p.rpc;
    a.tpr = p.tpr;
    a.heavy_links = p.heavy_links;
    a.list_cap = p.list_cap;
    a.blocked = p.blocked;
    a.hb_tpr = p.hb_tpr;
}

// Host-side launchers implemented in the .cu files.
// zbytes in {1,2,4}; returns a cudaError_t as int.
int launch_sweep(const SweepArgs& a, int zbytes, int rule, bool smem, int blocks, int threads,
                 size_t shared_bytes, void* stream);
int launch_energy(const EnergyArgs& a, void* stream);
// Time-sliced cooperative launch of `grid` blocks (state in shared memory);
// with grid = 0 it only reports the resident blocks per SM in *blocks_per_sm.
int launch_sweep_sliced(const SweepArgs& a, int zbytes, int rule, int grid, int threads, size_t shared_bytes,
                        void* stream, int* blocks_per_sm);
// Persistent batched kernel; set_attr = false during stream capture.
int launch_batch(const BatchArgs& b, int is_float, int kind, int zbytes, int rule, bool smem, int blocks,
                 int threads, size_t shared_bytes, void* stream, bool set_attr);
int sweep_max_shared_optin();
// Persistent serving kernel (blocks of rpc * tpr threads; grid = 0 only sets
// the shared-memory attribute); returns a cudaError_t as int.
int launch_serve(const ServeArgs& s, int grid, size_t shared_bytes, void* stream);
// Static shared memory of the serving kernel (per block).
size_t serve_static_shared();

}  // namespace sa
