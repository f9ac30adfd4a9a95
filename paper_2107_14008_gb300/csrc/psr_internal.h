// Internal declarations shared by the host builder, the C ABI and the CUDA
// kernels of libpsr.  Not part of the public ABI (see include/psr.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "psr.h"

namespace psr {

// Positions are quantised to 21 bits per axis for the Morton order; leaf-cell
// centres are integers in units of L / 2^22 (a cell of level l and index i has
// its centre at (2i + 1) 2^(21 - l)), so centre differences, with a periodic
// shift of n * 2^22, are integers below 2^24 in magnitude and convert to FP32
// exactly.
constexpr int kMortonBits = 21;
constexpr int kCentreShift = 22;
constexpr int kMaxLeaf = 64;
constexpr int kShiftCodes = 27;  // (nx+1)*9 + (ny+1)*3 + (nz+1)
constexpr int kMaxTableN = 8192;
constexpr int kFineMaxN = 1024;      // intervals of PSR_FP32_EXACT's fine table
constexpr int kMaxTaylorN = 2048;    // Taylor tables: 32-byte entries
constexpr int kTaylorPaperN = 384;   // x_c / 384 = 3 / 512 at x_c = 2.25, the paper's spacing

// Kinds of launch with a rule of their own for the parts of rows (parts_rule):
// the FP32 forward and adjoint with the linear table and with others, FP64.
enum : int { kPartsFwd, kPartsFwdTab, kPartsAdj, kPartsAdjTab, kPartsF64, kPartsKinds };

// Per-box constants as the kernels see them (plain old data, 16B aligned).
struct alignas(16) BoxDev {
    double L, r_s, r_c, G;      // FP64 path
    double rc2, inv_2rs, pad0, pad1;
    float unit;     // (L / 2^22) / (2 r_s): centre units -> FP32 coordinate units
    float x_c;      // r_c / (2 r_s): cutoff in FP32 coordinate units (= x)
    float x_c2;     // x_c^2
    float g_acc;    // G / (2 r_s)^2: FP32 coordinate sums -> acceleration
    float g_adj;    // G / (8 r_s^3): adjoint position gradient factor
    float g_adjm;   // G / (4 r_s^2): adjoint mass gradient factor
    float m_eq;     // the mass every particle of the box has (as FP32), 0 if they differ
    float pad3;
    // rows of more than above[kind] evaluated pairs are summed in parts[kind] parts
    int64_t above[kPartsKinds];
    int parts[kPartsKinds], pad4;
};
static_assert(sizeof(BoxDev) == 160, "BoxDev layout");

// Byte offsets of the regions of the device workspace (256-byte aligned).
struct Layout {
    size_t pf;       // float4[n]    FP32 leaf-local coords / (2 r_s), mass
    size_t pd;       // double4[n]   FP64 wrapped coords, mass (optional)
    size_t perm;     // int32[n]     sorted -> original
    size_t leaf;     // int4[nl]     first, count, box, pad
    size_t lcen;     // int4[nl]     centre x, y, z (units L/2^22), level
    size_t rowptr;   // int64[nl+1]  CSR of pair entries by target leaf
    size_t pairs;    // uint32[np]   (source leaf << 5) | shift code
    size_t items;    // int32[nl]    target leaves in schedule order
    size_t cost;     // int64[nl]    evaluated pairs of each leaf's row
    size_t boxes;    // BoxDev[nbox]
    size_t table;    // float4[2 * (kMaxTableN + 1)]: T table, then exp(-x^2)
    size_t core;     // float2[kMaxTableN + 1]: core form of the forward's linear table
    size_t fine;     // float4[2 * (kFineMaxN + 1)]: PSR_FP32_EXACT's fine table of T, then exp(-x^2)
    size_t t64;      // double[2][6 (kPlain64MaxN + 1)]: FP64 plain path's T and exp(-x^2) tables
    size_t cotf;     // float4[n] / double4[n] adjoint source payload scratch
    size_t ctrl;     // uint32[64]  scheduler tickets, error word, counters
    // multipole split (device builds with an acceptance parameter only)
    size_t frow;     // int64[nl+1]  CSR of well-separated (M2L) entries by target leaf
    size_t fpairs;   // uint32[nf]   (source leaf << 5) | shift code
    size_t fcen;     // double4[nl]  expansion centre (particle box centre), radius
    size_t fofs;     // float4[nl]   that centre minus the cell centre (lcen), radius
    size_t total;
};

// ctrl word indices
enum : int {
    kCtrlTicketFwd = 0,
    kCtrlDoneFwd = 1,
    kCtrlTicketAdj = 2,
    kCtrlDoneAdj = 3,
    kCtrlError = 8,
    kCtrlPairsLo = 16,  // uint64 at words 16..17: pairs within the cutoff
    kCtrlEvalLo = 18,   // uint64 at words 18..19: pairs evaluated
    kCtrlHeavy = 32,    // words 32..35: heavy items of each level (heavy_cost)
    kCtrlWords = 64,
};
// error bits
enum : unsigned {
    kErrLeafIndex = 1u,
    kErrParticleRange = 2u,
    kErrItemIndex = 4u,
    kErrShiftCode = 8u,
    kErrParts = 32u,     // a row of more parts than its group has warps
    kErrLookback = 16u,  // a look-back of the device build's scans or sorts ran out
};

// What a table region of the workspace holds: the table (key) and its x_c, put
// there by a launch that was enqueued (capture 0) or recorded under stream
// capture (capture: 1 + its id); and which table the graphs' replays write.
struct TableState {
    int key = -1;
    double x_c = -1.0;
    unsigned long long capture = 0;
    int recorded = -1;  // -1 none, -2 several
};

struct Leaves {
    int nbox = 0;
    std::vector<psr_box> boxes;
    std::vector<BoxDev> boxdev;
    std::vector<int64_t> box_first;  // first particle of each box (original numbering)
    int64_t n = 0;
    int max_leaf_req = 0;
    int flags = 0;
    double build_seconds = 0.0;
    // sorted particles
    std::vector<float> pf;     // 4 per particle
    std::vector<double> pd;    // 4 per particle
    std::vector<int32_t> perm32;
    std::vector<int64_t> perm;
    // leaves
    std::vector<int32_t> leaf;  // 4 per leaf
    std::vector<int32_t> lcen;  // 4 per leaf
    std::vector<int64_t> rowptr;
    std::vector<uint32_t> pairs;
    std::vector<int32_t> items;
    std::vector<int64_t> cost;       // evaluated pairs of each leaf's row
    std::vector<int64_t> item_cost;  // the same in schedule order
    int32_t n_heavy[4] = {0, 0, 0, 0};  // host copy of ctrl[kCtrlHeavy..] (psr_upload)
    int64_t evaluated = 0;
    int64_t max_cost = 0;  // the largest leaf's evaluated pairs
    int max_leaf = 0;
    int max_row = 0;
    // counts (set by both builders; a device-built handle has no host arrays)
    int64_t n_leaves = 0;
    int64_t n_pairs = 0;
    bool has_pd = false;        // FP64 payload present in the workspace
    bool device_built = false;  // arrays were built on the device
    bool equal_mass = false;    // in every box all particles share one mass (BoxDev::m_eq)
    bool has_far = false;       // pair list split into P2P (near) and M2L (far) entries
    double theta = 0.0;         //   multipole acceptance parameter of that split
    int64_t n_far = 0;          //   far entries
    char* db_scratch = nullptr; // device build between its two calls: the caller's scratch
    int db_kslot = 0;           //   runs per row in the pair cache (0: not used)
    int64_t db_uncached = 0;    //   and the rows it could not hold
    int64_t db_redo = 0;        //   rows to be walked again
    // device state
    Layout lay{};
    char* d_ws = nullptr;
    size_t ws_bytes = 0;
    bool uploaded = false;
    TableState table, core, fine, t64;  // what the workspace's table regions hold
    int sm_count = 0;
    int device = -1;
};

// builder.cpp
int build_batch(int nbox, const double* const* pos, const double* const* mass, const int64_t* n,
                const psr_box* boxes, int max_leaf, int flags, Leaves** out, std::string* err);
Layout make_layout(const Leaves& h);
size_t table_entry_bytes(int interp);  // p2p_fwd_f32.cu
BoxDev box_constants(const psr_box& b);  // per-box kernel constants

// Heavy rows.  Where a launch's largest row exceeds a warp's share of the work, a
// row on one warp outlasts the others, or the chip is never filled: such rows
// are summed in parts, which a group of warps forms side by side.  The parts are
// a matter of the arithmetic (each is summed by itself, and the parts are added in
// order), so the rule looks at the row and its box alone: a box gives the same
// forces, bit for bit, in a batch and alone, in a shard and whole, whatever the
// launch's shape.  Whether warps form the parts side by side or one warp forms
// them in turn is up to the launch (group_rule).

// Work of a row above which it is heavy, at level l: 1/2, 1, 2 and 4 times a warp's
// share with 32 warps per SM.
constexpr int kHeavyLevels = 4;
constexpr int kPartsSms = 152;  // the chip the parts are meant for
inline int64_t heavy_cost(int level, int64_t evaluated)
{
    return (evaluated << level) / (64 * (int64_t)kPartsSms);
}

// The parts of a set's heavy rows when `warps` warps share its work, and the level
// of heavy_cost above which rows are heavy (-1: all are).  No parts unless the
// largest row exceeds `line` / 8 of a share; below it the largest-first order
// hides the longest row, and the group phase's registers cost 1-3 % (128^3 NFW in
// leaves of up to 64: 9.53 -> 9.66 ms).  Rows above about half a share are heavy,
// all of them when there are fewer leaves than warps, and the parts are as many
// (2, 4 or 8) as bring the largest row's to 3/2 of a share, with at least 2500
// pairs in a part (the group's barriers and the row's start-up latency cost about
// as much as 1500).  Forward, one warp per row against this: 5000 uniform
// particles 0.235 -> 0.081 ms, 32^3 0.28 -> 0.12, 110,000 NFW 2.57 -> 1.1, 64^3 NFW
// 2.3 -> 1.5; adjoint 32^3 0.28 -> 0.20.  Eight parts wherever there are any: 60,000
// uniform in leaves of up to 16 0.28 ms against 0.17 with two and 0.19 with none.
struct SplitRule {
    int parts, level;
};
inline SplitRule split_rule(int64_t max_cost, int64_t evaluated, int64_t n_leaves, int64_t warps, int line)
{
    SplitRule r{1, -1};
    const int64_t share = evaluated / (warps > 0 ? warps : 1);
    if (max_cost <= line * share / 8) return r;
    while (r.parts < 8 && 2 * max_cost > 3 * r.parts * share && max_cost >= 5000 * r.parts) r.parts *= 2;
    if (n_leaves >= warps)
        for (r.level = 0; r.level + 1 < kHeavyLevels && 3 * heavy_cost(r.level, evaluated) < share;)
            ++r.level;
    return r;
}

// The line of a kind of launch: 3/2 of a share; 5/4 where a pair costs more, as
// with every table but the linear one (cubic adjoint, 150,000 NFW 4.33 -> 2.72 ms
// against a line of 2), and 2 for the linear adjoint of leaves of up to 32, whose
// rows are short against the group's overheads (150,000 NFW in leaves of up to 16
// 1.95 ms, 2.05 with 3/2; 64^3 NFW 2.74 and 2.83; in leaves of up to 64, 512,000 NFW
// gain 5.96 -> 5.36 with 3/2).
inline int split_line(int kind, int max_leaf)
{
    return kind == kPartsAdj ? (max_leaf <= 32 ? 16 : 12) : kind == kPartsFwd ? 12 : 10;
}

// A box's parts, for each kind as a launch of that kind on the box alone has them:
// 32, 24 and 16 warps per SM for the FP32 forward, the FP32 adjoint and FP64.
inline SplitRule box_rule(int kind, int64_t max_cost, int64_t evaluated, int64_t n_leaves, int max_leaf)
{
    const int warps = kind == kPartsFwd || kind == kPartsFwdTab ? 32 : kind == kPartsF64 ? 16 : 24;
    return split_rule(max_cost, evaluated, n_leaves, (int64_t)kPartsSms * warps, split_line(kind, max_leaf));
}
inline void parts_rule(int64_t max_cost, int64_t evaluated, int64_t n_leaves, int max_leaf, BoxDev* b)
{
    for (int k = 0; k < kPartsKinds; ++k) {
        const SplitRule r = box_rule(k, max_cost, evaluated, n_leaves, max_leaf);
        b->parts[k] = r.parts;
        b->above[k] = r.level < 0 ? -1 : heavy_cost(r.level, evaluated);
    }
}

// How a launch takes rows with parts: there are none; groups of warps form them side
// by side; one warp forms them in turn.
enum : int { kRowsWhole = 0, kRowsJoint = 1, kRowsInTurn = 2 };

// kernels (launchers defined in the .cu files; return cudaError_t as int)
struct FwdArgs {
    const void* pf;
    const void* pd;
    const int32_t* perm;
    const int32_t* leaf;
    const int32_t* lcen;
    const int64_t* rowptr;
    const uint32_t* pairs;
    const int32_t* items;
    const BoxDev* boxes;
    const void* table;   // float4[(table_n + 1)] forward, then Q table
    unsigned* ctrl;
    const void* cot;     // adjoint: cotangent, original order
    void* cot_sorted;    // adjoint: sorted payload scratch
    void* out;           // forward: acc; adjoint: grad pos
    void* out_m;         // adjoint: grad mass (may be null)
    int64_t n;
    int64_t n_leaves;
    int64_t n_pairs;
    int n_items;
    int nbox;
    int table_n;
    int interp;
    int accum;
    int fold_every;
    int count_pairs;
    int warps_per_block;
    int blocks;
    int max_leaf;
    int variant;     // FP32 forward: PSR_KERNEL_SCALAR, _PACKED or _PAPER
    int stage_cap;   // FP32 kernels: staged particles per warp
    int item_stride; // this launch takes schedule entries ticket * stride + offset
    int item_offset;
    int t64_max;       // FP64 kernels: last node of the table
    const long long* cost;  // evaluated pairs of each row
    int rows;          // kRowsWhole, kRowsJoint or kRowsInTurn
    int kind;          // whose parts rows have (kParts...)
    const int* heavy;  // kRowsJoint: how many items groups of warps take (null: all)
    int group;         //   and the warps per group (divides warps_per_block)
    int fine;        // PSR_FP32_EXACT by the fine cubic table (interp and table_n are its)
    int core;        // FP32 forward: a.table is the core form of the linear table
    int equal_mass;  // every box has one particle mass: the FP32 kernels take it out of the sums
};

int launch_table(int table_n, int interp, double x_c, void* d_out, void* d_q_out, void* stream);
int launch_core_table(int table_n, double x_c, void* d_out, void* stream);
bool fwd_core(int precision, int interp, int table_n, int variant, double x_c);
int launch_fwd_f32(const FwdArgs& a, int precision, void* stream);
int launch_fwd_f64(const FwdArgs& a, double x_c, void* stream);
int launch_adj_f32(const FwdArgs& a, int precision, void* stream);
int launch_adj_f64(const FwdArgs& a, double x_c, void* stream);
int fwd_f32_occupancy(int precision, int interp, int accum, int warps, int table_n, int cap,
                      int variant, int core, int* out);
size_t fwd_f32_smem(int precision, int interp, int table_n, int warps, int cap);
constexpr size_t kSmemPerBlock = 227 * 1024;  // opt-in dynamic shared memory per block
int fwd_f64_occupancy(int warps, int interp, int table_n, double x_c, int* out);
int launch_table64(int table_n, int interp, double x_c, void* d_out, void* stream);  // p2p_fwd_f64.cu
size_t fwd_f64_smem(int interp, int table_n, double x_c, int warps);
// Nodes of the FP64 plain path's tables, per unit of x: a power of two, so that
// a distance in node spacings has the rounding of 1 / (2 r_s) alone.  The last
// node, x = 5.32, is what the allocation-free entry point's scratch holds; tail:
// the cutoff lies beyond it.
constexpr int kPlain64PerX = 256, kPlain64MaxN = 1363;
struct Plain64 {
    int n;
    bool tail;
};
Plain64 plain64(double x_c);
int launch_plain64(double x_c, void* d_t, void* d_q, void* stream);
int adj_f64_occupancy(int warps, double x_c, int* out);
size_t adj_f64_smem(double x_c, int warps);
int launch_fwd_blk(const FwdArgs& a, int precision, void* stream);  // p2p_fwd_blk.cu
int fwd_blk_occupancy(int precision, int interp, int accum, int max_leaf, int table_n, int* out);
int adj_f32_occupancy(int precision, int interp, int accum, int warps, int max_leaf, int table_n,
                      int cap, int variant, int* out);
size_t adj_f32_smem(int precision, int interp, int table_n, int warps, int cap);

}  // namespace psr
