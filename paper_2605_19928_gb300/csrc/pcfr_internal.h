// Internal layout shared by the host tree builder, the C ABI and the CUDA kernels.
//
// HBM layout (per subgame; every per-hand row is padded to `hstride` elements, a multiple
// of 32, so each row starts at least 128-byte aligned).  V is the value type: a pair of
// FP32 (hi, lo) in the default precision, or one FP32.
//   R, S         FP64 [n_rows][hstride]       cumulative regret / average-strategy sums
//   sigma        V    [n_rows][hstride]       current strategy (regret matching of R)
//   sigbar       V    [n_rows][hstride]       average strategy (exploitability pass)
//   reach        V    [2][n_nodes][hstride]   reach of each player under sigma
//   reach_bar    V    [2][n_nodes][hstride]   reach under the average strategy
//   cfv, cfv_br  V    [2][n_nodes][hstride]   counterfactual values (last traversal / BR)
// A decision node with A actions owns rows [row, row + A); player 0's rows come first.
//
// Terminal tables, one block of uint16 per showdown board (TermTab gives the offsets), all
// indices below 2^15 because a player has at most kMaxHands hands:
//   clh    [k * H]   per-card lists of hands, each list in rank-sorted order, concatenated
//   cards  [H]       card ids of each hand, c1 | c2 << 8 (c2 = 255 for one-card hands)
//   cloff  [deck+1]  start of each card's list in clh
//   perm   [H]       hand at each rank-sorted position
//   gs, ge [H]       first / one-past-last sorted position of each hand's tie group
//   lo, hi [2 * H]   per (hand, card) the clh index of the first entry at or after gs / ge
// Fold nodes need only the first three (board 0); the block is padded to 16 bytes so that
// the terminal kernel can stage it with one bulk (TMA) copy.
#pragma once
#include <cstddef>
#include <cstdint>

#ifndef __CUDACC__  // host-only translation units share the small helpers below
#define __host__
#define __device__
struct uint4 {
  uint32_t x, y, z, w;
};
#endif

namespace pcfr {

enum NodeType : uint8_t { kDecision = 0, kFold = 1, kShowdown = 2, kChance = 3, kLeaf = 4 };
// Fold, showdown and depth-limit leaf nodes: their values come from outside the per-hand
// tree passes (terminal and leaf launches).
__host__ __device__ inline bool is_end(int type) { return type == kFold || type == kShowdown || type == kLeaf; }

constexpr int kMaxActions = 16;
constexpr int kMaxHands = 1176;  // of a player: two of the 49 cards that a flop leaves
constexpr int kMaxDeck = 52;
constexpr uint8_t kNoCard = 255;
constexpr int kPrecisionPairs = 0;   // values as double-float FP32 pairs
constexpr int kPrecisionSingle = 1;  // values as FP32
constexpr int kDiscountCapacity = 1 << 11;  // iterations a new handle's discount table covers
                                            // (doubled on demand)
// Passes of the per-hand kernel (and of the wide schedule).
enum HandMode { kModeInit = 0, kModeUpdate = 1, kModeAvg = 2, kModeBR = 3 };

constexpr int kScheduleLevel = 1;   // per-hand passes: one block per chunk of hands, level by level
constexpr int kScheduleStream = 2;  // update pass: one warp per 32 hands walks a depth-first program
constexpr int kScheduleWide = 3;    // one large tree: every pass is a launch per level over all of
                                    // that level's (node, hand) pairs
constexpr int kStreamMaxActions = 8;  // actions at a decision node the stream schedule holds in registers
constexpr int kStreamHalfMin = 12;   // 8-byte units per lane in each half of a warp's prefetch ring,
                                      // at least (or the most one node needs, 2 A + 1)
constexpr int kStreamWarps = 4;       // warps per block of the stream schedule (one game per block)

struct alignas(16) NodeDev {
  int32_t parent;     // -1 at the root
  int32_t first_kid;  // children are consecutive: [first_kid, first_kid + n_kids)
  int32_t row;        // decision: first row; showdown: board table; otherwise -1
  int32_t arow;       // row of the action that leads here (parent's row + paction), or -1
  uint8_t type;       // NodeType
  uint8_t player;     // decision: acting player; fold: folding player
  uint8_t n_kids;
  uint8_t deal;       // card dealt by the chance parent, else kNoCard
  uint8_t paction;    // index among the parent's children
  uint8_t level;
  uint8_t aplayer;    // player acting at the parent decision, else kNoCard
  uint8_t pad;
  uint64_t board;     // public cards at this node (bit c = card c)
};
static_assert(sizeof(NodeDev) == 32, "NodeDev is 32 bytes");

// Hand tiles (k_tile): the table of one subgame, one block of uint16 staged in shared memory.
// Offsets are in uint16 from its start.
struct TileHead {
  int32_t inner;      // TileNode [n_inner]: inner nodes, level by level
  int32_t level;      // [levels + 1] first inner node of each level
  int32_t levels;     // levels that hold inner nodes
  int32_t ends, n_ends;        // node ids of the fold, showdown and leaf nodes
  int32_t rows[2];             // per player: TileRow of each of its rows
  // per player: the nodes that make new reach rows (TileNode whose id is the node holding the reach
  // at it, HostGame::reach_row), level by level; first of each level; levels
  int32_t fwd[2], flevel[2], flevels[2];
  int32_t all[2];              // per player: [n_nodes] reach_row
  int32_t deal;                // uint8 [n_nodes] card dealt to each node (none without chance nodes)
};
static_assert(sizeof(TileHead) % 16 == 0, "the table's TileNodes start 16-byte aligned");
// One inner node of a tile table, 8 bytes.
struct alignas(8) TileNode {
  uint16_t id, first_kid, row;  // row: of the node's first action, from its player's first row
  uint8_t kids;                 // children | (player, or 2 for a chance node) << 6
  uint8_t pad;
};
static_assert(sizeof(TileNode) == sizeof(uint64_t), "TileNode is 8 bytes");
struct alignas(8) TileRow {  // a row's child node, its decision node, and the node holding the reach there
  uint16_t kid, node, src, pad;
};

constexpr int kTileSmemSmall = 26 * 1024;  // shared memory of a block of 128 threads: eight fit an SM
constexpr int kTileSmem = 53 * 1024;       // of a block of 256 threads: four fit
constexpr int kTileSmemStaged = 200 * 1024;  // of the latency form, at most

// One node of the stream schedule's program (pre-order), 16 bytes.  Offsets are in
// elements of a per-hand array (multiples of hstride).
struct alignas(16) ProgOp {
  int32_t node_off;   // node * hstride
  int32_t row_off;    // decision: first row * hstride; otherwise 0
  uint32_t code;      // type (2 bits) | player << 2 | n_kids << 3 (6 bits) | deal << 9 (8 bits) |
                      // terminal-children mask << 17 (bit a: child a is a fold or showdown;
                      // chance nodes: bit 0, all children are)
  int32_t first_kid;
};

// One load of the stream schedule's prefetch: array << kArrShift | element offset.
enum StreamArray : uint32_t { kArrR = 0, kArrS = 1, kArrReach = 2, kArrCfv = 3, kArrM = 4 };
constexpr uint32_t kArrShift = 29, kArrOffMask = (1u << 29) - 1u;
static_assert(sizeof(ProgOp) == 16, "ProgOp is 16 bytes");

// Offsets (in uint16) of the terminal-table sections for H hands of k cards from a deck.
struct TermTab {
  int clh, cards, cloff, fold_len, perm, gs, ge, lo, hi, len;
  __host__ __device__ static int round8(int x) { return (x + 7) / 8 * 8; }
  __host__ __device__ TermTab(int H, int k, int deck) {
    clh = 0;
    cards = k * H;
    cloff = cards + H;
    fold_len = round8(cloff + deck + 1);
    perm = fold_len;
    gs = perm + H;
    ge = gs + H;
    lo = ge + H;
    hi = lo + 2 * H;
    len = round8(hi + 2 * H);
  }
};

// Everything one subgame's kernels need: read-only tables and the solver state.
struct GameDev {
  int n_nodes, n_levels, n_hands, hstride, hand_size, n_rows, n_terminals, deck;
  int chunk, n_chunks;  // hands per block in the per-hand passes
  int smem;             // per-hand pass keeps its chunk's state in shared memory (the same
                        // for every game of a handle)
  int row_begin[3];     // player p owns rows [row_begin[p], row_begin[p + 1])
  int n_boards;
  double kappa64;              // 1 / Z, Z = sum of r0(h0) r1(h1) over hand pairs sharing no card
  const NodeDev* nodes;
  const double* payoff;        // [n_nodes] terminal payoff magnitude times the probability of
                               // the public cards dealt on the path (fold: folder's chips in,
                               // showdown: each player's chips in); 0 elsewhere
  const float* payoff_ff;      // [n_nodes][2] payoff * kappa64 as an FP32 pair (hi, lo), rounded
                               // once on the host: the terminal scale (FP32 values use hi)
  const int32_t* level_start;  // [n_levels + 1]
  const int32_t* row_node;     // [n_rows] decision node owning each row
  const int32_t* dec_nodes;    // decision nodes of player 0, then of player 1
  int dec_begin[3];            // player p's are dec_nodes[dec_begin[p] .. dec_begin[p + 1])
  const uint64_t* hand_mask;   // [n_hands]
  const void* range_v;         // [2][hstride] normalised ranges, value type V
  const double* range64;       // [2][hstride]
  const uint16_t* term_tab;    // [n_boards][TermTab.len]
  const uint4* term_rec;       // [n_boards][n_hands] (grouped terminal launch): cards, gs, ge, then lo and
                               // hi per card, as uint16
  const ProgOp* prog;          // [prog_len] inner nodes in depth-first pre-order (stream schedule)
  int prog_len;
  const uint16_t* tile_tab;    // hand tiles: TileHead and its lists (null: the handle does not use them)
  int tile_tab16;              // its length in 16-byte units
  int tile_wlog;               // log2 of the hands per tile
  int tile_group;              // threads that walk its levels in the latency form and k_resident
  const int32_t* chunks;       // load chunks of the stream schedule (see stream_tables)
  int chunk_off[4], chunk_count[4];
  const uint32_t* units;       // loads of the stream schedule, in the order the passes use them
  int unit_off[4], unit_count[4];
  // state
  double* R;
  double* S;
  double* M;                   // Predictive CFR+ prediction [n_rows][hstride] (else null)
  void* sigma;
  void* sigbar;
  void* reach;
  void* reach_bar;
  void* cfv;
  void* cfv_br;
  uint64_t* xval;              // resident schedule, alternating: stamped values [2][n_nodes][hstride][sizeof(V) / 4]
  uint64_t* xreach;            // and stamped reach rows, laid out alike
  double* br_partial;          // [2][n_chunks] per-block sums of r_i(h) v*_i(root, h)
  double* br_out;              // [2]
  unsigned* br_done;           // blocks of the best-response pass that have finished
};

struct PairF {  // an FP32 pair: a value hi + lo
  float hi, lo;
};

// Per player, the node whose reach row stands for a terminal's (HostGame::reach_row), negated and
// less one (~node) where the hands holding a card dealt since are to be zeroed.
struct TermSrc {
  int32_t row[2];
};
__host__ __device__ inline int term_src_node(int32_t row) { return row < 0 ? ~row : row; }

// Up to four terminal nodes of one game, board table and kind, evaluated together (FP32 values).
struct alignas(16) TermGroup {
  int32_t game;
  int32_t table;      // board table (folds read table 0)
  int16_t kind;       // kFold or kShowdown
  int16_t count;
  int32_t below;      // bit p: player p's reach at some node is another's without dealt cards' hands
  int32_t node[4];
  TermSrc src[4];
  uint64_t board[4];
  float pay[2][4];    // per player: payoff * kappa, negative where the player folded
};
static_assert(sizeof(TermGroup) == 128, "TermGroup is 128 bytes");
constexpr int kTermSegment = 32;  // groups a block of the grouped terminal launch walks at most

// Wide schedule: an inner node, and a node that makes a new reach row of one player.
struct alignas(16) WideNode {
  uint32_t id;        // node | children << 24 | (player, or 2 for a chance node) << 30
  int32_t first_kid;
  int32_t row;        // decision: first row
  int32_t src;        // decision: node whose reach row of its player stands for its own
  __host__ __device__ int node() const { return (int)(id & 0xffffffu); }
  __host__ __device__ int kids() const { return (int)(id >> 24 & 63u); }
  __host__ __device__ int kind() const { return (int)(id >> 30); }
};
struct alignas(16) WideReach {
  int32_t node, src;  // src: node whose row it derives from (-1: the root, from the range)
  int32_t arow;       // row of the player's action that leads here, or -1
  int32_t deal;       // dealt card, or -1
};

struct Work {
  int game;
  int unit;  // chunk index (per-hand passes) or node id (terminal pass)
};

// Per-iteration update weights for iteration t (entry t - 1): DCFR's positive / negative
// regret discounts and average discount, and the weight of the new average contribution.
struct Discount {
  double dpos, dneg, dS, wS;
};

// Kernel entry points (kernels.cu), all asynchronous on `stream`.
struct LaunchCtx {
  const GameDev* games;        // device array
  int n_games;
  const Work* chunk_work;      // device [n_chunk_work]: (game, chunk)
  int n_chunk_work;
  const Work* term_work;       // device [n_term_work]: (game, terminal node), grouped by game,
                               // board table and kind (folds, then showdowns)
  int n_term_work;
  int term_nv;                 // nodes a block evaluates together: 1 (in runs when n_term_runs > 0), or
                               // term_groups of up to 2 or 4
  const TermGroup* term_groups;   // device (term_nv > 1)
  const Work* term_runs;       // device [n_term_runs]: (first entry of term_work, count), one block's (run form)
  int n_term_runs;
  bool term_swap;              // run form: scan arrays with entries swapped within eights
  const Work* term_segments;      // device [n_term_segments]: (first group, count), one block's
  int n_term_segments;
  const TermSrc* term_src;     // device [n_term_work]: reach rows of each terminal
  const int32_t* reach_row[2]; // device [n_nodes] (run-out tables): HostGame::reach_row
  int* iter;                   // device: iterations completed
  unsigned* done;              // device: block arrival counter
  int* err;                    // device: nonzero after a bounded wait gave up
  const Discount* disc;        // device [iterations covered], one entry per iteration
  size_t smem_hand;            // dynamic shared memory of the per-hand kernel; 0 = every game
                               // works on the global arrays (some tree is too large to stage)
  size_t smem_term;            // dynamic shared memory of the terminal kernel
  int variant;
  int precision;               // kPrecisionPairs or kPrecisionSingle
  int pdl;                     // chain launches with programmatic dependent launch
  int schedule;                // kScheduleLevel, kScheduleStream (update launches) or kScheduleWide
  const Work* warp_work;       // device [n_warp_work]: (game, first group of 32 hands) of each
                               // block of the stream schedule, largest trees first
  int n_warp_work;
  const Work* tile_work;       // device [n_tile_work]: (game, tile), largest trees first; the per-hand
  int n_tile_work;             // passes run as k_tile when there are any
  size_t smem_tile;            // dynamic shared memory of k_tile
  int tile_threads;            // its threads per block
  int tile_staged;             // its latency form (R and S staged; level and wide schedules)
  int stream_depth;            // stack slots per lane of the stream schedule
  int stream_prog;             // nodes of the largest tree, if its program is staged in shared
                               // memory; 0 = read from global memory
  int stream_half;             // units per lane in each half of the stream prefetch ring
  int stream_units;            // load descriptors staged per block (0 when the program is not)
  int stream_hp;               // hands per lane of the stream schedule (1 or 2): a warp owns 32 * stream_hp
  // wide schedule (one game): level l's inner nodes are wide_inner[wide_inner_off[l] ..
  // wide_inner_off[l + 1]); per player, the nodes that make new reach rows at depth d (0: the root) are
  // wide_fwd[p][wide_fwd_off[p][d] .. wide_fwd_off[p][d + 1])
  int wide_levels;             // number of levels
  const int* wide_inner_off;   // host [wide_levels + 1]
  const WideNode* wide_inner;  // device, level by level
  int wide_fwd_levels[2];
  const int* wide_fwd_off[2];  // host [wide_fwd_levels + 1]
  const WideReach* wide_fwd[2];  // device
  int wide_pairs;              // pairs of hands: a thread takes one
  int wide_segments;           // k_wide_back: blocks per node, and
  int wide_threads;            // threads of each
  int wide_max_dec;            // decision nodes of the player who has more
  // resident schedule (cfr_iterate only; the other passes use the level schedule's kernels)
  int resident;                // cfr_iterate runs k_resident
  int resident_grid;           // blocks of the cooperative launch (>= n_chunk_work)
  size_t smem_resident;        // its dynamic shared memory: terminal region, then hand region
  unsigned resident_term;      // bytes of the terminal region
  bool resident_ahead;         // some tree's regrets are matched ahead of the walk (with pairs)
  unsigned* resident_sync;     // device [3]: barrier arrivals, blocks finished (zero between launches), the last stamp used
  int alternating;
};

int launch_init(const LaunchCtx& c, void* stream);
int launch_terminal(const LaunchCtx& c, int player_mask, int use_bar, void* stream);
int launch_update(const LaunchCtx& c, int player_mask, int advance, void* stream);  // either schedule
int launch_current_rows(const LaunchCtx& c, void* stream);  // sigma = RM(R), every game (read-back)
int launch_avg_reach(const LaunchCtx& c, void* stream);
int launch_br(const LaunchCtx& c, void* stream);
int launch_average_rows(const LaunchCtx& c, void* stream);
// Kernels one pass of the wide schedule launches (which: kModeInit, kModeUpdate, kModeAvg or
// kModeBR, as the per-hand kernel's modes).
int wide_launch_count(const LaunchCtx& c, int which, int player_mask, int advance);
int hand_kernel_smem_limit();
// Shared memory of one block of the terminal launch for one game (nv: LaunchCtx::term_nv; runs: its run form).
// Whether a thread's run of either scan of the run form is a multiple of eight entries.
bool scans_in_eights(int n_hands, int hand_size, size_t es);
size_t terminal_smem_size(int n_hands, int hand_size, int deck, int hstride, size_t es, int nv, bool runs);
// Shared memory the per-hand kernel needs to stage one game (es = bytes per value).
size_t hand_smem_size(int n_nodes, int n_levels, int rows_max, int W, size_t es);
int configure_kernels();  // once per process, before the first launch
// Polls of the terminal kernel's first bulk-copy wait on the current device (< 0: the
// default limit); for tests of the timeout path.  Returns 0 or -1.
int set_first_wait_polls(long polls);
// Shared memory of k_tile for one game (tab16: its table in 16-byte units; staged: its latency form).
size_t tile_smem_size(int tab16, int n_nodes, int rows_max, int W, size_t es, int staged);
// Resident schedule: shared memory of its two regions for one game, the blocks of k_resident
// one SM holds with `smem` bytes (0 if none), and the cooperative launch of n_iters iterations.
size_t resident_term_size(int n_hands, int hand_size, int deck, int hstride, size_t es);
size_t resident_hand_size(int tab16, int n_nodes, int rows_max, int W, size_t es);
int resident_blocks_per_sm(int precision, size_t smem);
int launch_resident(const LaunchCtx& c, int n_iters, void* stream);
// Dense layer of the leaf network (leafnet.cu): C[M][N] = act(A[M][K] B[N][K]^T + bias), BF16
// A and B, FP32 accumulation, C in BF16 (out_f32 = 0) or FP32; N a multiple of 128, K of 64.
// Returns 0, -1 (launch failed), -2 (bad shape or alignment), -3 (no tensor-map encoder).
int launch_gemm_bf16(const void* A, const void* B, const float* bias, void* C, int M, int N, int K, int act,
                     int out_f32, int* err, void* stream);
int configure_gemm();

// ---- depth-limit leaf network (leafnet.cu)
// Network input per (leaf, river card): both players' reach at the leaf over the 1326
// two-card slots (each normalised to sum 1 over the hands not holding the river card), a
// one-hot of the 5 board cards, then 2 pot / stack features; zero padding to kLeafIn.
// Output: each player's value per unit pot over the 1326 slots; padding to kLeafOut.
constexpr int kLeafSlots = 1326;
constexpr int kLeafFeatures = 2 * kLeafSlots + 52 + 2;  // 2706
constexpr int kLeafIn = 2752;                           // padded to a multiple of 64
constexpr int kLeafHidden = 512;
constexpr int kLeafOut = 2688;                          // 2 x 1326 padded to a multiple of 128
constexpr int kLeafCards = 48;                          // river cards after 4 board cards

struct LeafDev {      // one depth-limit leaf
  int game, node;
  int src[2];         // per player, the node whose reach row stands for the leaf's
  int row0;           // first of its kLeafCards network rows (river cards ascending)
  float feat[2];      // pot / (pot + 2 stack), stack / (pot + 2 stack) at the leaf
};

struct LeafCtx {
  const LeafDev* leaves;   // device [n_leaves]
  int n_leaves;
  const int16_t* slot;     // per game [hstride]: slot of each hand (device, game-major)
  const int16_t* hand_at;  // per game [kLeafSlots]: hand in each slot or -1
  int hstride_max;
  void* X;                 // [rows][kLeafIn] BF16
  void* H1;                // [rows][kLeafHidden] BF16
  void* H2;
  void* H3;
  float* Y;                // [rows][kLeafOut]
  const void* W[4];        // BF16 [out][in]
  const float* b[4];
  int hand_order;          // 1: every game has the same hand list, and the network's range
                           // inputs and value outputs are laid out in that list's order
                           // (hand h at column h of each player's 1326) -- the first and last
                           // layers' weights are permuted to match -- so the leaf kernels
                           // read and write them coalesced; 0: slot order
};

// The network's input rows (use_bar: of the average strategy), its four layers -- the last for the
// outputs of player 0, player 1 or both (mask 1, 2, 3) -- and the leaf values of player i (use_bar:
// into cfv_br).  launch_leaf_outputs is the last layer alone, from the hidden rows L.H3.
int launch_leaf_inputs(const LaunchCtx& c, const LeafCtx& L, int use_bar, void* stream);
int launch_leaf_net(const LaunchCtx& c, const LeafCtx& L, int player_mask, void* stream);
int launch_leaf_outputs(const LaunchCtx& c, const LeafCtx& L, int player_mask, void* stream);
int launch_leaf_values(const LaunchCtx& c, const LeafCtx& L, int player, int use_bar, void* stream);
// Dynamic shared memory of one stream-schedule block: the staged program (prog_nodes nodes)
// and one player's load descriptors (prog_units), and per lane a prefetch ring of 2 x half
// units of hp 8-byte entries and a stack of `depth` slots of hp values (es bytes each).
inline size_t stream_smem_size(int prog_nodes, int prog_units, int half, int depth, size_t es, int hp) {
  return (size_t)prog_nodes * sizeof(ProgOp) + (size_t)prog_units * 4 +
         (size_t)kStreamWarps * 32 * hp * (2 * (size_t)half * 8 + (size_t)depth * es);
}

}  // namespace pcfr
