// pt_kernels.cuh -- launch arguments of the build, walk and force stages
// (internal to libpt.so).
#pragma once

#include "pt_internal.cuh"

struct pt_ctx;

namespace pt {

constexpr unsigned kWalkStackSmall = 768;    // per-warp walk stack entries (shared memory)
constexpr unsigned kWalkStackLarge = 12288;  // retry size after an overflow
constexpr unsigned kOrbitStack = 2048;       // per-warp stack of the orbit-dependent search
constexpr unsigned kWalkMaxIters = 1u << 24;   // safety cap on walk iterations per group
constexpr unsigned long long kWalkChunkEntries = 8192;   // one-pass list allocation granule

// A group is wide when a side of its grid box is at least 2^-kWalkWideShift of
// the root box: it is listed by the build and walked by a whole block (see
// pt_walk.cu).  2^-4 finds the groups with many times the mean list (a box
// that reaches the core from the halo) among 9 to 1% of a Plummer sphere's
// groups (16,384 to 250,007 particles); 2^-5 lists twice as many at the same
// walk times.  In uniform sets nearly every group is wide up to 10^5 particles,
// and their walks are no slower for it (one warp per group -> now: sphere of
// 16,384 102 -> 72 us, of 100,003 204 -> 167, of 250,007 319 -> 294; cube of
// 100,003 211 -> 168; a fractal of 100,003 143 -> 90).  Sets below
// kWalkWideMin particles have none: their walks take a few dozen steps, and a
// block's steps cost more than a warp's (1,000 particles: 39 against 32 us).
constexpr unsigned kWalkWideShift = 4, kWalkWideMin = 2048;
__device__ __forceinline__ bool walk_wide(const uint4 ga, const uint4 gb, unsigned set_n) {
    return set_n >= kWalkWideMin && max(max(gb.x - ga.x, gb.y - ga.y), gb.z - ga.z) >= (kGrid >> kWalkWideShift);
}

struct BuildArgs {
    unsigned n;                      // particles (all sets)
    const unsigned *n_dev;           // device copy of n
    int nsets;
    const double *pos, *mass;        // input order (device)
    SetInfo *sets;                   // nsets
    unsigned *set_of;                // n (only when nsets > 1)
    unsigned long long *bmin, *bmax; // 3 * nsets
    unsigned long long *keys_in;     // n
    unsigned *vals_in;               // n
    uint4 *qbuf;                     // n
    unsigned long long *skey;        // n
    unsigned *perm;                  // n
    double4 *sp64;
    float4 *spH, *spL;
    uint4 *sq;
    // nodes
    unsigned cap_nodes;
    uint4 *nd_a, *nd_b;
    uint2 *nd_r;
    double4 *nd_c, *nd_q, *nd_t;
    float4 *nd_f;
    uint4 *nd_bnd;                   // 2 per node: child boundaries of split nodes (build only)
    unsigned *nd_int;                // per level from lvl_begin: its internal nodes (build only)
    unsigned *topo_bsum;             // children counted per block of the topology grid (build only)
    unsigned char *lcp;              // n + 32 bytes: shared key digits of neighbours (build only)
    unsigned *tmp_u32a, *tmp_u32b;   // max(cap_nodes, n) each
    // groups
    unsigned *gflag, *gbegin;        // n each
    uint2 *gr_r;
    uint4 *gr_a, *gr_b;
    unsigned *gr_wide;               // groups with a wide box, in any order
    int n_leaf, n_group;
    // deepest level the launch sequence covers (kMaxLevel: every tree): the
    // depth of a recent build of the tree plus a margin (two at first, doubled
    // whenever a tree was deeper, so that one that often is ends at every
    // level), since an empty level still costs its three kernels; a deeper
    // tree is flagged (kErrLevels) and built again.  Not used by sets small
    // enough for one block (kSmallBuild in pt_build.cu)
    int levels;
    // mass-dependent changeover radii (Eq. 12): per-particle factors in input
    // order (NULL: computed from the masses when massdep, else all 1)
    const double *scale;
    int massdep;
    double *scale_buf;               // n (device-computed factors)
    double *set_mean;                // nsets
    double *ssc;                     // n, sorted factors
    long long *nd_thr, *gr_thr;      // gap thresholds per node / group
    Status *status;
    ScanTmp scan_tmp;
    SortTmp sort_tmp;
};

struct WalkArgs {
    const uint4 *nd_a, *nd_b;
    const uint2 *nd_r;
    const uint2 *gr_r;
    const uint4 *gr_a, *gr_b;
    const unsigned *gr_wide;             // groups walked by whole blocks, in any order
    const SetInfo *sets;
    const long long *nd_thr, *gr_thr;    // per node / group gap thresholds (massdep)
    int massdep;
    WalkParams wp;
    unsigned *gr_nc, *gr_np;
    unsigned long long *gr_co, *gr_po;   // ngroups + 1
    // PP entries of leaves whose box is at least r_out from the group's box
    // (opened for the opening angle only: no pair within r_out), kept apart
    unsigned *gr_nf;
    unsigned long long *gr_fo;
    unsigned *cells, *pp;
    unsigned long long cap_cells, cap_pp;
    unsigned long long chunk_cells, chunk_pp;   // one-pass allocation granules (entries)
    unsigned stack_cap;                  // stack entries per warp
    unsigned *spill;                     // per-warp spill areas of the stack (global memory)
    unsigned spill_cap;                  // entries per warp in the spill area
    Status *st;
    ScanTmp scan_tmp;
};

struct ForceArgs {
    const uint2 *gr_r;
    const uint4 *gr_a, *gr_b;        // group grid boxes (qmin, set), (qmax, -)
    const unsigned *gr_nc, *gr_np;
    const unsigned long long *gr_co, *gr_po;
    const unsigned *gr_nf;           // far PP segment (no pair within r_out)
    const unsigned long long *gr_fo;
    // work items, written per launch by k_items_write in processing order: (group,
    // part | parts << 16); groups of more than one part also have a slot in gr_pb
    // (index of their first partial record, parts finished)
    uint2 *items;
    uint2 *gr_pb;
    unsigned *item_bsum;             // items per block and class (8 per SM)
    double4 *parts;                  // partial sums: part_stride targets per record
    unsigned part_stride;
    unsigned item_cap, part_cap;     // items the launch can take, records in parts
    unsigned part_shift;             // scale of the part length by precision: see part_entries
    const unsigned *cells, *pp;
    const double4 *sp64;
    const float4 *spH, *spL;
    const double4 *nd_c, *nd_q;
    const float4 *nd_f;
    const uint2 *nd_r;
    const uint4 *sq;
    float4 *ffp, *ffn;               // float64 kernel: float32 expansions (4 per particle, 7 per node)
    const SetInfo *sets;
    const unsigned *perm;
    const double *ssc;               // sorted radius factors (massdep)
    int massdep;
    double *acc, *pot;               // input (caller) order, device
    double G;
    double theta;                    // opening angle of the lists
    int order;                       // 0 or 2
    int want_nb;
    uint2 *pairs;                    // (sorted i, sorted j)
    unsigned long long pair_cap;
    // CTAs of the launch, each first taking the item of its own index.  The
    // item count is on the device: a single set's grid holds the group count
    // (known after the build) and the extra parts of the last step with head
    // room, and a step that needs more is flagged and repeated; a batch's
    // grid is a hint from its previous step (count_hint = 1: items beyond
    // the grid go to CTAs that take them from an atomic counter).  0: a
    // persistent launch taking every item from the counter.
    unsigned direct_items;
    unsigned count_hint;
    double4 *gpart;                  // per group: sum m phi / 2, sum m a
    double4 *red_e;                  // per reduction block: partial sums of gpart
    unsigned long long *red_c;       // per reduction block: cell and PP interaction counts
    Status *st;
};

struct NbArgs {
    unsigned n;                      // particles (all sets)
    const unsigned *perm;
    const uint2 *pairs;
    unsigned long long pair_cap;
    unsigned *npairs_dev;            // clamped pair count (device)
    unsigned long long *keys, *keys_sorted;
    unsigned *vals, *vals_sorted;
    long long *nb_off;               // n + 1 (global CSR, input order)
    int *nb_idx;                     // pair_cap
    int key_bits;
    unsigned *row;                   // n: entries per row
    const unsigned *n_dev;           // device copy of n
    Status *st;
    ScanTmp scan_tmp;
    SortTmp sort_tmp;
};

// Orbit-dependent neighbour search (Sec. 6.3.1, Eq. 24) on a built tree.
struct OrbitArgs {
    unsigned n;
    const unsigned *perm;
    const double4 *sp64;
    const float4 *spH, *spL;             // float-float split of the sorted positions
    const uint4 *sq;
    const double *ssc;
    int massdep;
    const SetInfo *sets;
    const uint4 *nd_a, *nd_b;
    const uint2 *nd_r;
    const uint2 *gr_r;
    const uint4 *gr_a, *gr_b;
    const double *vel;                   // input order, n x 3 (device)
    double dt, C_r, C_v, G;
    int mode;                            // 0 r_out reference, 1 r_nb reference, 2 candidates
    double4 *sv;                         // sorted (v, r_nb)
    float *rnbf;                         // sorted r_nb as float (prefilter)
    double *nd_rnb;                      // per node: largest r_nb
    long long *nd_thr, *gr_thr;          // gap thresholds from r_nb
    double *rnb_out;                     // optional: r_nb in input order
    uint2 *pairs;
    unsigned long long pair_cap;
    unsigned long long *ctr;             // [0] work counter, [1] candidates
    unsigned stack_cap;
    unsigned cap_nodes;
    const unsigned *gr_wide;             // wide groups
    int max_level;                       // deepest level of the tree
    Status *st;
};
int orbit_launch(const OrbitArgs &A, cudaStream_t st);

// Per-set pointer table of a batch (device resident).
struct BatchTab {
    const double *pos, *mass;
    const double *scale;             // radius factors or NULL
    double *acc, *pot;
    long long *nb_off;
    int *nb_idx;
    unsigned long long nb_cap;
};

int batch_gather_launch(const BatchTab *tab, const SetInfo *sets, int nsets, unsigned n,
                        double *pos, double *mass, double *scale, cudaStream_t st);
int batch_scatter_launch(const BatchTab *tab, const SetInfo *sets, int nsets, unsigned n,
                         const double *acc, const double *pot, cudaStream_t st);
int batch_nb_launch(const BatchTab *tab, const SetInfo *sets, int nsets, unsigned n,
                    const long long *off, const int *idx, long long *totals, bool split,
                    cudaStream_t st);
int build_launch(const BuildArgs &A, cudaStream_t st);   // returns kernels launched
int walk_init();   // once per context: kernel attributes of the walk
// Context access for the auxiliary entry points outside pt_api.cu: selects the
// context's device and returns its stream; ctx_fail records a message.
cudaStream_t ctx_enter(pt_ctx *ctx);
int ctx_fail(pt_ctx *ctx, int code, const char *msg);
int walk_warps(unsigned stack_cap);   // warps of a walk launch with this stack size
constexpr unsigned kWalkSpill = 4096;    // per-warp spill entries of the walk stack (global memory)
int walk_launch(const WalkArgs &A, int phase, cudaStream_t st);    // 0 count+scan, 1 fill, 2 one pass
int force_launch(const ForceArgs &A, int precision, unsigned n, cudaStream_t st);
constexpr unsigned kForce64Unit = 128;    // list entries of one tile of every warp of the float64 kernel
int force64_launch(const ForceArgs &A, unsigned n, int blocks, cudaStream_t st);
constexpr int kRedBlocksMax = 256;    // partial-sum slots of the force's energy / momentum reduction
int force_reduce_launch(const ForceArgs &A, cudaStream_t st);
constexpr unsigned kNbRowMax = 512;   // longest neighbour row nb_launch sorts (else: status max_row above it)
int nb_launch(const NbArgs &A, cudaStream_t st);
int nb_sort_launch(const NbArgs &A, cudaStream_t st);   // rows of any length

}  // namespace pt
