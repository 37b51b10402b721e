// Internal data structures shared by the host compiler/runtime and the CUDA
// kernels.  Plain structs only (no STL) so that device code can read them.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define VL_HD_INLINE __host__ __device__ __forceinline__
#else
#define VL_HD_INLINE inline
#endif

namespace vl {

// ----------------------------------------------------------------- geometry
// Bit-packed masks: Wp = 4 * ceil(W / 128) words per row, LSB first.
static inline int words_per_row(int w) { return ((w + 127) / 128) * 4; }

// Connected-component tiles: up to CCL_TH rows x CCL_TWW words (1024 px),
// labelled as CCL_NS strips of two rows; one lane owns a 32-px word.
constexpr int CCL_TH = 32;
constexpr int CCL_TWW = 32;
constexpr int CCL_NS = CCL_TH / 2;
// A strip run can start at every column under 4-adjacency (checkerboard).
constexpr int CCL_MAXRUNS = CCL_NS * CCL_TWW * 32;

// Components of a tile that reach its border: at most one per row-run start
// of the first and the last row and per pixel of the outer columns.
constexpr int CCL_MAXBORDER = 2 * CCL_TWW * 16 + 2 * CCL_TH;

constexpr int EXEC_THREADS = 512;  // threads per CTA of every tiled kernel
constexpr int EXEC_WARPS = EXEC_THREADS / 32;

// Buffers of a fused group: rows of 16-byte vectors, the tile's words and one
// vector left and right of them (vectors per row, bytes of one buffer).
VL_HD_INLINE int group_vecs(int tile_words) { return (tile_words + 3) / 4 + 2; }
static inline int64_t group_buffer_bytes(int rows, int tile_words) {
  return (int64_t)rows * group_vecs(tile_words) * 16;
}
// Shared memory in front of the buffers: instructions of a segment (and one
// behind them), and which of them are loads.
constexpr int GROUP_SEG = 256;
constexpr int64_t GROUP_PROG_BYTES = (GROUP_SEG + 1) * 16 + (GROUP_SEG + 8) * 2;
static_assert(GROUP_PROG_BYTES % 16 == 0, "buffers start on 16-byte boundaries");
// Shared memory the buffers of a context's largest tiles may take: 14
// buffers of a 32 x 32-word tile with 8 halo rows above and below.
constexpr int64_t kGroupBudget = 14 * 48 * 10 * 16;

// Device status word values (match vl_status where they overlap).
constexpr int ST_OK = 0;
constexpr int ST_TIMEOUT = 6;
constexpr int ST_INTERNAL = 8;
// Which consistency check failed (bits 8.. of the status word, with
// ST_INTERNAL in the low byte).
constexpr int RS_GFIND = 1 << 8;     // global find ran past its bound
constexpr int RS_GUNION = 2 << 8;    // global union ran past its bound
constexpr int RS_FLIST = 3 << 8;     // (unused: no flagged-root list any more)
constexpr int RS_TLOAD = 4 << 8;     // saved tile state out of range
constexpr int RS_TRUNS = 5 << 8;     // more strip runs than a tile holds
constexpr int RS_SUNION = 6 << 8;    // shared union-find ran past its bound
constexpr int RS_GRANGE = 7 << 8;    // global union-find entry outside the image
constexpr int RS_SELECT = 8 << 8;    // percentile select not down to one key

// --------------------------------------------------------- group bytecode
// One instruction of a fused tile group.  Buffers are shared-memory tiles of
// (th + 2*halo) rows x group_vecs vectors; `h` is the halo (in rows and
// pixels) over which this node's value is needed.
enum InsnOp : uint8_t {
  I_NOP = 0,
  I_THR = 1,     // dst = image[img].channel[ch] (> or <) t      (aux bit0: lt,
                 //   bit1: t comes from the job's percentile slot `slot`)
  I_LOAD = 2,    // dst = materialised mask slot `slot`
  I_NOT = 3,     // dst = not a
  I_AND = 4,     // dst = a and b
  I_OR = 5,      // dst = a or b
  I_NEAR = 6,    // dst = N a (connectivity of the formula)
  I_CONST = 7,   // dst = all-false (aux 0) or all-true (aux 1)
  I_STORE = 8,   // materialised mask slot `slot` = a   (core region only)
  I_ANDNOT = 9,  // dst = a and not b
  I_RTHR = 10,   // dst = threshold by rank code: table a, code bound K = img
                 //   (as uint16), code bits = ch, first plane = slot; aux
                 //   bit0: lt (see RankTab)
};

// Bit of Insn::op: a block barrier precedes the instruction (the compiler
// places one only where a thread may touch a buffer word that another
// thread touched since the previous barrier).
constexpr uint8_t I_SYNC = 0x80;

struct Insn {        // 16 bytes
  uint8_t op;        // InsnOp, with I_SYNC
  uint8_t dst;
  uint8_t a;
  uint8_t b;
  int16_t h;         // halo of this node within the group
  int16_t slot;      // materialised-mask slot / percentile slot
  int16_t img;       // image index (THR)
  int16_t ch;        // channel (THR)
  float t;           // threshold constant (THR)
};
static_assert(sizeof(Insn) == 16, "Insn layout");
VL_HD_INLINE int insn_op(const Insn& in) { return in.op & ~I_SYNC; }

// -------------------------------------------------------------- plan steps
enum StepKind : int32_t {
  SK_PCT = 0,        // percentile selects: one item per percentile slot
  SK_GROUP = 1,      // fused pointwise/N tile group: one item per tile
  SK_RZ_LOCAL = 2,   // rho batch, tile-local labelling + publish: item = (rz, tile)
  SK_RZ_MERGE = 3,   // rho batch, union across tile borders: item = (rz, chunk)
  SK_RZ_UNUSED = 4,  // (no longer emitted: the seed flag travels with the keys)
  SK_RZ_FINAL = 5,   // rho batch, relabel + write Z: item = (rz, tile)
  SK_RANK = 6,       // rank codes of threshold tables: item = (table, row block)
  SK_ARITH = 7,      // number terms: item = row block, writes the number images
  SK_PCT_PASS = 8,   // (on the device only: a pass of percentile selects,
                     //   item = (percentile slot, share of the channel); which
                     //   pass in `halo`)
};

// Rows of one arithmetic work item.
constexpr int ARITH_ROWS = 4;

// Number terms of a formula as one straight-line program run per pixel on a
// register file of floats: A_VALUE loads image[img].channel[ch], the
// operations read registers a and b (b = kArithConst: the constant c) and
// write dst, A_STORE writes register a to number image `img` (counted from
// the first number image).  Every operation rounds to float once.
enum ArithOp : uint8_t { A_VALUE = 0, A_ADD = 1, A_SUB = 2, A_MUL = 3, A_DIV = 4, A_STORE = 5 };
constexpr uint8_t kArithConst = 0xFF;
constexpr int kArithMaxRegs = 16;
constexpr int kArithMaxInsns = 1024;
struct ArithInsn {   // 12 bytes
  uint8_t op, dst, a, b;
  int16_t img, ch;
  float c;
};
static_assert(sizeof(ArithInsn) == 12, "ArithInsn layout");

// Rows of one rank-code work item.
constexpr int RANK_ROWS = 8;

// Percentile selects over many blocks: passes (one on the range a sample
// gives; three more, of 12 bits each, if that misses), words of a select in
// global memory, and how many blocks share a select when `side_by_side`
// selects run at once on `slots` resident blocks: enough to fill those,
// each with at least 8192 pixels (one round of its threads' loads).
constexpr int SEL_PASSES = 4;
constexpr int SEL_BINS = 4096;
constexpr int SEL_HIST = 16 + SEL_PASSES * SEL_BINS;
// Channels from which many blocks share a select (batch_build says why).
constexpr int64_t SEL_SPLIT_PIXELS = 1 << 18;
static inline int select_blocks(int64_t pixels, int64_t side_by_side, int64_t slots) {
  int64_t n = slots / side_by_side, most = (pixels + 8191) / 8192;
  if (n > most) n = most;
  return n < 1 ? 1 : (int)n;
}

struct StepDesc {
  int32_t kind;
  int32_t insn_off;  // groups: first instruction (into the formula's insns)
  int32_t insn_cnt;
  int32_t halo;      // groups: halo rows/px
  int32_t rz_off;    // rho batches: first RZ entry
  int32_t rz_cnt;
  int32_t pct_off;   // percentile step: first PCT entry
  int32_t pct_cnt;   // (groups, on the device: loads in pct_off, float thresholds in
                     //   pct_cnt among its instructions)
  int32_t rank_mask; // groups: rank tables (< 32) its I_RTHR read, one bit each
  int32_t rank_halo; // groups: largest halo of those I_RTHR
  int32_t n_bufs;    // groups: tile buffers its instructions use (0 .. n_bufs-1);
                     //   the shared-memory stage of rank planes follows them
};

// Rank codes of one image channel against the sorted distinct constant
// thresholds t_1 < ... < t_m of a formula on that channel: a pixel value v
// has code c = 2 * #{k : t_k < v} + [v equals some t_k] (0 for NaN), kept
// as `nbits` bit planes (bit b of every pixel's code in plane plane0 + b)
// plus a plane of NaN pixels (plane0 + nbits).  Then v > t_k exactly when
// c >= 2k, and v < t_k exactly when c < 2k - 1 and v is not NaN, so every
// threshold of the table becomes one bit-sliced comparison with a constant.
struct RankTab {
  int32_t img, ch;
  int32_t m;         // thresholds in the table
  int32_t nbits;     // code bits: bit length of 2m + 1
  int32_t val_off;   // first threshold value in the formula's value array
  int32_t plane0;    // first plane of the table in the job's plane array
};

// Component select Z = union of phi2-components meeting N phi1 (the core of
// rho, Sec. 3.2); the compiler lowers rho phi1[phi2] to N(phi1 or Z).
struct RzDesc {
  int16_t phi1_slot;
  int16_t phi2_slot;
  int16_t z_slot;
  int16_t scratch;   // index of the job's CCL scratch set used
};

struct PctDesc {
  int16_t img;
  int16_t ch;
  int16_t slot;      // percentile slot written
  int16_t pad;
  double q;
};

// ----------------------------------------------------- executor job table
// Pixel formats of number images.
constexpr int32_t PX_F32 = 0;
constexpr int32_t PX_U16 = 1;

struct DevImage {
  const void* data;        // number images: channels planes of H x pitch
                           //   elements (float, or uint16 by `format`)
  const uint32_t* mask;    // mask images: H x Wp words
  int32_t channels;
  int32_t is_mask;
  int32_t format;          // PX_F32 or PX_U16
  int32_t written;         // 1: written earlier in the same launch (number
                           //   images of SK_ARITH): read through L2, not the
                           //   read-only path
};

struct DevJob {
  int32_t H, W, Wp, pitch;      // pitch in floats = 32 * Wp
  int32_t n_steps;
  int32_t step_base;            // into the launch's step table
  int32_t gth, gtww;            // group tile rows / words
  int32_t g_tiles_y, g_tiles_x; // group tiles
  int32_t c_tiles_y, c_tiles_x; // CCL tiles
  int32_t conn;
  int32_t n_images;
  const DevImage* images;
  uint32_t* const* slots;       // materialised mask slots: the intermediate
                                // ones back to back at slot_mem, the roots'
                                // at root_mem, then those of mask images
  uint32_t* slot_mem;
  uint32_t* root_mem;
  int32_t n_inter_slots, n_root_slots;
  const Insn* insns;
  const RzDesc* rz;
  const PctDesc* pct;
  float* pct_val;               // percentile values by slot
  uint32_t* sel_hist;           // state of the percentile selects (SEL_HIST words
                                //   each), null: a select is one block's work
  // CCL scratch sets, one per select of a batch step, `set_bytes` apart:
  // union-find over keys (G, 2 * H * W entries: pixel ids and the keys of
  // unseeded components), saved tile state (tiles x tile_cap words)
  unsigned char* rzs;
  int64_t set_bytes;
  int64_t off_state;
  int32_t tile_cap;
  int32_t c_th;                 // rows of a labelling tile (16 or 32)
  int32_t* status;              // device status word of this job
  const RankTab* rtab;          // rank tables of the formula
  const float* rvals;           //   their sorted threshold values
  int32_t n_rtab;
  int32_t sel_blocks;           // blocks that share a percentile select
  uint32_t* planes;             // rank-code planes, H x Wp words each
  const ArithInsn* arith;       // number-term program (SK_ARITH)
  int32_t n_arith;
  int32_t arith_regs;           //   registers it uses
  int32_t first_num_image;      // image index of number image 0
  int32_t pad_;
};

VL_HD_INLINE int32_t* rz_G(const DevJob& J, int k) {
  return reinterpret_cast<int32_t*>(J.rzs + k * J.set_bytes);
}
VL_HD_INLINE int32_t* rz_state(const DevJob& J, int k) {
  return reinterpret_cast<int32_t*>(J.rzs + k * J.set_bytes + J.off_state);
}

// A step of a job as the executor takes it up, in one load of a warp: what it
// is, and which steps (of the launch) it waits for until they have done how
// many sub-items.
constexpr int REC_DEPS = 8;
struct StepRec {
  StepDesc step;
  int32_t per_rz;      // rho batches: sub-items of each
  int32_t n_deps;
  int32_t more;        // dependencies beyond REC_DEPS: the first, in the launch's list
  int32_t pad[2];
  struct Dep { int32_t step, need; } dep[REC_DEPS];
};
static_assert(sizeof(StepRec) == 128, "a word per lane");

// One work item of the persistent executor: a range of `count` consecutive
// sub-items (tiles, chunks, rz x tile) of one step of one job.
struct WorkItem {
  int32_t job;
  int32_t step;        // step index within the job; on the device, of the launch
  int32_t first;       // first sub-item
  int32_t count;       // sub-items in this item
};

}  // namespace vl
