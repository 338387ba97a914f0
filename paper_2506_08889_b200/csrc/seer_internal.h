// Host-side declarations shared by the translation units of the library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace seer {

constexpr int kHeadDim = 128;       // d
constexpr int kTileTokens = 64;     // tokens per staged K (or V) tile
constexpr int kMaxGroup = 8;        // query heads per KV head handled by one MMA N-tile
constexpr int kMaxDGate = 256;      // gate width: 64, 128 or 256
constexpr int kMaxRounds = 12;      // halving rounds of the decode kernels' dynamic tile pool

// Kernel attributes (the opt-in to more dynamic shared memory) are per device: index of the current
// device into per-device "already configured" tables (processes here use one GPU, the library does
// not assume it).
constexpr int kMaxDevices = 64;
inline int current_device_slot() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
    return dev % kMaxDevices;
}

// Launch with the programmatic-stream-serialisation attribute (see pdl_wait in seer_device.cuh).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// Everything the decode kernels need besides the two tensor maps.
struct DecodeParams {
    const __nv_bfloat16* q;
    __nv_bfloat16* out;
    float* lse;
    const int32_t* seq_lens;
    const int32_t* block_idx;       // sparse only
    const int32_t* block_cnt;       // sparse only, may be null
    const int32_t* page_table;      // paged only
    int64_t page_table_stride;
    int max_sel;
    int page_size;
    int num_pages;
    int batch, num_q_heads, num_kv_heads, group, block_size, tiles_per_block;
    int blocks_per_tile;            // 64 / block_size for blocks of 16 or 32 tokens (a tile gathers several listed blocks), else 1
    int bs_shift, tpb_shift, bpt_shift;   // log2 of block_size, tiles_per_block, blocks_per_tile
    unsigned int kvh_magic;         // ceil(2^32 / num_kv_heads), 0 for one KV head: unit / num_kv_heads by __umulhi
    int group_magic;                // ceil(2^16 / group): r / group = (r * group_magic) >> 16 for r < 64
    int q_len;                      // query tokens per sequence (the last q_len cached tokens), 1 for plain decoding
    int t_base, t_cnt;              // this launch handles query tokens t_base .. t_base + t_cnt - 1
    int rows;                       // t_cnt * group: rows on the MMA N side, <= 8 * (N-tiles of the kernel)
    int num_units;                  // batch * num_kv_heads
    int max_blocks_cap;             // tile-count clamp for dense: capacity in tiles
    int pool_div;                   // 1/pool_div of the tiles are handed out dynamically (0: none)
    int min_tiles;                  // a CTA's range has at least this many tiles (fewer CTAs take part when work is short)
    int max_rounds;                 // most dynamic chunks per range (<= kMaxRounds; 0: none) -- bounds the partial slots
    float scale_log2;               // sm_scale * log2(e)
    const int* list_flags;          // non-null: unit u's list is final once list_flags[u] == list_gen (written by the gate
    int list_gen;                   // kernel of the same step); the producer warp then waits per unit, not for the gate's grid
    int sel_from_lens;              // > 0: every unit's list holds min(this, blocks of its sequence) entries, so the
                                    // counts follow from the lengths and the schedule can be made before the kernel
                                    // that writes the lists has finished (0: read block_cnt)
    int next_early;                     // cluster kernels: StepPlan's, ListPlan's
    int clusters;                       // list kernel: ListPlan's
    int spread;                         // list kernel: ListPlan's (sel_from_lens > 0: behind a step that has done even lists itself)
    unsigned int* status;
    unsigned long long* tickets;    // [num_units]: tiles done << 32 | valid-slot bits; zero between launches
    int* sched;                     // [2]: theft cursor, exit counter; zero between launches
    int* steal;                     // [grid]: per-range claim counters (front | back << 16); zero between launches
    unsigned int generation;        // stamp that marks this launch's partials
    int* prefix;                    // [num_units + 1] prefix sums of the units' tile counts
    float* part_o;                  // [slots][8*NT][128]   (NT: N-tiles of the kernel, 1 or 2)
    float* part_ml;                 // [slots][32*NT]: max[8*NT], sum[8*NT], generation stamp
#ifdef SEER_DECODE_TRACE
    unsigned long long* trace;      // [grid][8] %globaltimer stamps (diagnostic builds only)
#endif
};

struct DecodeLaunch {
    int grid;
    cudaStream_t stream;
};

// Returns resident CTAs per SM for the decode kernel (queried once).
int decode_ctas_per_sm(bool sparse, bool paged, int n_tiles);
// Upper bound on the number of work intervals (static ranges + dynamic chunks) of a launch.
int decode_max_intervals(int grid, int max_rounds = kMaxRounds);
// n_tiles: MMA N-tiles of 8 rows (1 or 2: tokens on M), or 8 for the variant with the unit's (up to 64) rows on M;
// p.rows <= 8 * n_tiles.
cudaError_t launch_decode(bool sparse, bool paged, int n_tiles, const CUtensorMap& map_k, const CUtensorMap& map_v,
                          const DecodeParams& p, int grid, cudaStream_t stream);

struct GateParams {
    const __nv_bfloat16* q_nope;    // [B,Hq,d]
    const __nv_bfloat16* w_q;       // [Hkv,dg,g*d]
    const __nv_bfloat16* kcomp;     // [B,Hkv,max_blocks,dg]
    const int32_t* seq_lens;
    const float* scores_in;         // may be null
    float* scores;                  // [B,Hkv,max_blocks] (workspace or caller's scores_out)
    float* scores_user;             // caller's scores_out or null
    float* q_gate;                  // [B,Hkv,dg] workspace
    int32_t* block_idx;
    int32_t* block_cnt;
    int batch, num_q_heads, num_kv_heads, group, block_size;
    int d_gate, max_blocks, max_sel, token_budget;
    int q_len;                      // query tokens per sequence (1 for plain decoding); q_nope is [B,q_len,Hq,d]
    int threshold_mode;             // 0: token budget, 1: softmax probability above `threshold`
    float threshold;
    unsigned int* status;
    int* tickets;                   // [B*Hkv], zero between launches
    // One-launch step: the block that has just filled, if any, is compressed in the same launch (see KcompParams).
    const __nv_bfloat16* k_nope;    // null: no append
    const __nv_bfloat16* w_k;
    int64_t k_stride_batch, k_stride_head, k_stride_token;
    int k_rows_block_local;
    int* list_flags;                // non-null: list_gen is stored (release) to list_flags[u] once unit u's list is written
    int list_gen;
    double inv_freq[kMaxDGate / 2]; // rope_theta^(-2c/d_gate), computed on the host in double
};
// The one-kernel form of short calls (seer_step.cu): one cluster of S CTAs per unit.
constexpr int kStepMaxBlocks = 16384;   // compressed keys per unit that its gate holds in shared memory
// How a call of `units` units of `rows` (query token, head) rows whose lists are at most max_tiles tiles long runs as one
// launch.  With the gate: max_keys compressed keys per unit, max_codes tiles or, if these are smaller, blocks per unit;
// else 0.  (max_tiles = 0: the gate alone.)
struct StepPlan {
    int S;                              // CTAs per cluster; 0: not a short call
    int parts, rows;                    // clusters per unit, which have `rows` of its rows each (the last one the rest)
    bool wide;                          // 16 worker warps per CTA, one CTA per SM (else 8 and two)
    bool next_early;                    // the stream's next launch may start beside this one
    bool spread;                        // a step whose lists may be so long that it matters whether they are even: the list kernel, with
                                        // as many CTAs per unit, comes behind it
};
StepPlan step_plan(int units, int rows, int q_len, long long max_tiles, long long max_codes, int max_keys);
// g == nullptr: attention only (of several query tokens), over p.block_idx (nullptr: all blocks).  p.q == nullptr: the gate only.
cudaError_t launch_step_cluster(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g,
                                const StepPlan& plan, cudaStream_t stream);
// One query token over given lists, or all blocks, as one launch of a cluster of S CTAs per unit (seer_lists.cu).
constexpr int kListTiles = 128;         // most tiles a CTA
constexpr int kListUnits = 320;         // most units whose tiles it counts
struct ListPlan {
    int S;                              // CTAs per cluster; 0: the decode kernel
    int clusters;                       // one per unit, and more where units are few and long
    bool spread;                        // the lists may be so long that it matters whether they are even
    bool next_early;                    // the stream's next launch may start beside this one
};
ListPlan list_plan(int units, long long max_tiles);
// Bytes of partial results (DecodeParams::part_o) that a launch may need.
size_t list_part_bytes(int units, int clusters, int S);
cudaError_t launch_lists(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, int S, cudaStream_t stream);
// The gate by itself as one launch of such clusters (at most 8192 compressed keys per unit), while they are resident all at
// once; false: not that size, and nothing has been launched.
bool launch_gate_cluster(const GateParams& p, cudaStream_t stream, cudaError_t* err);
// Launches the scoring kernels (unless scores_in is given) and the selection kernel.
// Returns the number of kernels launched through *launched.
cudaError_t launch_gate_select(const GateParams& p, cudaStream_t stream, int* launched);
// Whether a gate over max_blocks compressed keys per unit runs as the one cluster kernel (the only
// path that takes several query tokens).
bool gate_one_kernel(int max_blocks);

struct KcompParams {
    const __nv_bfloat16* k_nope;
    const __nv_bfloat16* w_k;       // [Hkv,dg,3d]
    __nv_bfloat16* kcomp;           // [B,Hkv,max_blocks,dg]
    const int32_t* seq_lens;
    int64_t stride_batch, stride_head, stride_token;
    int rows_block_local;
    int first_block, num_blocks;    // first_block == -t (1..8): the block that filled while the last t tokens were appended
    int wait_at_end;                // append only: work first, wait for the preceding kernel just before the end
    int batch, num_kv_heads, block_size, d_gate, max_blocks;
    int sm_count;                   // bulk build: one persistent CTA per SM
    unsigned int* status;           // sticky device status word (bounded waits report here)
#ifdef SEER_DECODE_TRACE
    unsigned long long* trace;      // diagnostic builds: per-warp cycle counters of the bulk build
#endif
    double inv_freq[kMaxDGate / 2];
};
// True when the bulk build of these parameters runs as the persistent streaming kernel, which reads the keys
// through a tensor map (channel, token row, head, sequence) with a box of 64 channels x kKcompStageRows rows (or a
// block's, if it has fewer), 128-byte swizzle; launch_kcomp_append falls back to the plain-load kernel when it is given
// no map.
constexpr int kKcompStageRows = 64;
bool kcomp_bulk_streams(const KcompParams& p);
cudaError_t launch_kcomp_append(const KcompParams& p, const CUtensorMap* map_k, cudaStream_t stream, int* launched);

}  // namespace seer
