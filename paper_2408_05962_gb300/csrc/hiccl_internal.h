// Internal data structures shared by the host factorizer (hiccl_plan.cpp) and
// the device runtime (hiccl_runtime.cu).  Not part of the public ABI.
#pragma once

#include <algorithm>
#include <cstdint>
#include <new>
#include <string>
#include <vector>

#include "../../include/hiccl.h"

#ifdef __CUDACC__
#define HICCL_HD __host__ __device__
#else
#define HICCL_HD
#endif

namespace hiccl {

// ---------------------------------------------------------------------------
// device-side layout of an uploaded plan
// ---------------------------------------------------------------------------

// A warp moves one segment of a step at a time: at most SEG_BYTES of every
// operand (the staging slot size).  FP8 steps use segments of whole 144-byte
// blocks.
constexpr uint32_t SEG_BYTES = 4096;
constexpr uint32_t FP8_BLOCK_ELEMS = 128;
constexpr uint32_t FP8_BLOCK_BYTES = 144;   // 128 e4m3 codes, binary32 scale, 12 zero bytes
HICCL_HD inline uint32_t seg_bytes_of(uint32_t dtype) { return dtype == 3u ? 28u * FP8_BLOCK_BYTES : SEG_BYTES; }
constexpr uint32_t MAX_ENTRIES_PER_ITEM = 64;
// executor CTAs assumed when a plan is made without a device to query: a
// 152-SM GB300 at two CTAs per SM
constexpr unsigned long long DEFAULT_GRID = 304;
// work-item sizing (measured on the seven collectives of 4 MiB per rank at
// P = 64): pipeline slots under SMALL_SLOT_BYTES are spread over the grid,
// larger ones over LARGE_SLOT_ITEMS items
constexpr unsigned long long SMALL_SLOT_BYTES = 12ull << 20;
constexpr unsigned long long LARGE_SLOT_ITEMS = 768;
constexpr uint32_t MAX_FANIN = 1024;    // reduce inputs / copy destinations per step
constexpr uint32_t TMA_MAX_FANIN = 8;   // reduce inputs folded in shared memory

enum : uint32_t { OP_COPY = 0, OP_REDUCE = 1 };

// meta word of a step: op (2 bits) | dtype (4) | aligned16 (1) | reduction
// operator (3) | nsrc (11) | ndst (11)
HICCL_HD inline uint32_t meta_pack(uint32_t op, uint32_t dt, uint32_t al, uint32_t nsrc, uint32_t ndst,
                                   uint32_t rop = 0) {
  return op | (dt << 2) | (al << 6) | (rop << 7) | (nsrc << 10) | (ndst << 21);
}
HICCL_HD inline uint32_t meta_op(uint32_t m) { return m & 3u; }
HICCL_HD inline uint32_t meta_dtype(uint32_t m) { return (m >> 2) & 15u; }
HICCL_HD inline uint32_t meta_aligned(uint32_t m) { return (m >> 6) & 1u; }
HICCL_HD inline uint32_t meta_rop(uint32_t m) { return (m >> 7) & 7u; }
HICCL_HD inline uint32_t meta_nsrc(uint32_t m) { return (m >> 10) & 2047u; }
HICCL_HD inline uint32_t meta_ndst(uint32_t m) { return (m >> 21) & 2047u; }

// one contiguous run of a step's segments inside a work item
struct DevEntry {
  uint32_t step;
  uint32_t seg_lo;
  uint32_t seg_hi;
  uint32_t pad;
};

// A run of an item: consecutive entries whose steps have identical shape and
// operands that continue one another in memory (adjacent pipeline channels of
// one branch), moved as one range.  `entry` is the run's first entry within
// the item; `off` the byte offset in that entry's step where the run starts.
struct DevRun {
  uint32_t entry;
  uint32_t pad;
  unsigned long long off;
  unsigned long long bytes;
};

// ---- work-item records ----------------------------------------------------
// Everything the control warp stages for one work item lies in one contiguous,
// 16-byte aligned record, brought into shared memory by bulk copies in a
// single round trip: the entries (step, meta word, pointer offset, dependency
// count), the prefix sums of the runs' segment counts, the runs, and the
// operand pointers of the entries' steps.  A pointer offset with PTR_GLOBAL
// set indexes the global pointer array instead (steps with many operands, or
// an item whose inline pointer area is full).
constexpr uint32_t PTR_CAP = 160;              // inline pointers per item
constexpr uint32_t SUCC_CAP = 128;             // inline successors per item
constexpr uint32_t SUCC_GLOBAL = 0xffffffffu;  // the item's successor lists stay global
constexpr uint32_t PTR_STEP_MAX = 64;          // a step with more operands keeps them global
constexpr uint32_t PTR_GLOBAL = 0x80000000u;
struct RecEnt {
  uint32_t step;
  uint32_t meta;
  uint32_t poff;    // inline pointer index, or PTR_GLOBAL | global pointer index
  uint32_t indeg;   // dependency count of the step
};
struct DevItem {
  uint32_t rec;     // record offset in 16-byte units
  uint32_t nent;
  uint32_t nrun;
  uint32_t nptr;    // inline pointers
  uint32_t nsucc;   // inline successors, or SUCC_GLOBAL
  uint32_t pad[3];
};
static_assert(sizeof(RecEnt) == 16 && sizeof(DevItem) == 32 && sizeof(DevRun) == 24, "record layout");
HICCL_HD inline uint32_t rec_ent_bytes(uint32_t nent) { return nent * 16u; }
HICCL_HD inline uint32_t rec_rpre_bytes(uint32_t nrun) { return ((nrun + 1u) * 4u + 15u) & ~15u; }
HICCL_HD inline uint32_t rec_run_bytes(uint32_t nrun) { return (nrun * 24u + 15u) & ~15u; }
HICCL_HD inline uint32_t rec_ptr_bytes(uint32_t nptr) { return (nptr * 8u + 15u) & ~15u; }
// completion section: per entry the step's completion target, then the
// offsets of the entries' successor lists (nent + 1), then the successors
HICCL_HD inline uint32_t rec_cmp_words(uint32_t nent, uint32_t nsucc) {
  return 2u * nent + 1u + (nsucc == SUCC_GLOBAL ? 0u : nsucc);
}
HICCL_HD inline uint32_t rec_cmp_bytes(uint32_t nent, uint32_t nsucc) { return (rec_cmp_words(nent, nsucc) * 4u + 15u) & ~15u; }
HICCL_HD inline uint32_t rec_bytes(const DevItem &it) {
  return rec_ent_bytes(it.nent) + rec_rpre_bytes(it.nrun) + rec_run_bytes(it.nrun) + rec_ptr_bytes(it.nptr) +
         rec_cmp_bytes(it.nent, it.nsucc);
}

// control block (device memory, zeroed at upload).  Work items are claimed
// from one ticket counter that is never reset between launches: launch e
// (from 0) makes exactly nitems + grid claims (every CTA claims until it
// draws a ticket past the last item), so ticket t belongs to launch
// t / (nitems + grid) and names item t mod (nitems + grid).  The launch index
// scales the dependency targets; no CTA does any work at exit.
struct DevCtl {
  unsigned long long ticket;   // claims so far, over all launches
  unsigned long long err;      // nonzero: abort (code << 32 | step)
};

struct DevTable {
  const unsigned char *recs;          // work-item records (16-byte aligned)
  const DevItem *items;               // [nitems] record descriptors, in ticket order
  const uint32_t *nent;               // [nsteps] entries covering the step (completion target)
  const uint32_t *succ_off;           // [nsteps + 1]
  const uint32_t *succ;               // [nedges]
  const unsigned long long *ptrs;     // [nptrs] device addresses (nsrc sources then ndst destinations per step)
  unsigned long long *dep;            // [nsteps] arrivals of predecessors (cumulative over launches)
  unsigned long long *done;           // [nsteps] finished entries (cumulative over launches)
  DevCtl *ctl;
  unsigned long long *host_err;       // mapped host word mirroring ctl->err
  unsigned long long nitems;
  unsigned long long timeout_ns;
  unsigned long long seg;             // segment bytes of this plan
  unsigned long long *trace;          // [nitems][6] timestamps, SM, first step; or null (see hiccl_get_trace)
};

enum : uint32_t { ERR_TIMEOUT = 1, ERR_BADSTEP = 2, ERR_STALL = 3 };

// ---- sweeps -------------------------------------------------------------------
// A program whose primitives form independent expressions over equal byte
// ranges runs as one pass over its outputs instead of step by step: a
// *member* evaluates one expression -- a copy of one source, or the nested
// fold of several -- element by element and stores the value to every
// destination.  Partial sums stay in registers (rounded to the payload where
// the schedule's steps would round them) and no relay is written or read, so
// a pass moves each input and each output once.  Members of equal shape form
// a class; a class is cut into warp-sized units.
constexpr uint32_t SWEEP_SMS = 152;        // of a GB300 (plans are made without a device too)
constexpr uint32_t SWEEP_MAX_DEPTH = 6;    // partial values held while an inner group is folded
constexpr uint32_t SWEEP_PREFIX = 96;      // classes of a launch searched in the parameter bank
constexpr uint32_t SWEEP_INLINE = 4;       // classes of a launch passed as arguments

// kernel of a launch
enum : uint32_t {
  SWEEP_COPY = 0,     // copies whose operands lie equally far off a 16-byte boundary
  SWEEP_FOLD = 1,     // folds of such operands (and copies beside them), 32-bit or BF16 values
  SWEEP_FP8 = 2,      // folds of FP8 blocks
  SWEEP_NARROW = 3,   // folds of other operands: 4- or 2-byte accesses
  SWEEP_SHIFT = 4,    // copies of other operands: vectors shifted in registers
  SWEEP_TEAM = 5,     // folds as SWEEP_FOLD's, a CTA to a unit
  SWEEP_FP8_TEAM = 6, // folds as SWEEP_FP8's, a CTA to a unit
  SWEEP_KERNELS = 7
};
// A copy's destinations are stored in groups of SWEEP_GROUP, group after group
// over SWEEP_TILE / (vectors per lane) units of source (4 MiB, which stay in
// L2 between the groups): few, long streams of writes instead of one per
// destination.  Measured, 4 MiB to 64 destinations in turn over three sets of
// buffers: all 64 a unit 54 us, 16 44 us, 8 43 us, 4 40.7 us, 2 38.0 us
// (7.2 TB/s), 1 40.4 us.  16 MiB to 16 destinations by tiles of 1 / 2 / 4 / 8 /
// 16 MiB: 43.1 / 42.5 / 41.2 / 42.4 / 45.9 us.
constexpr uint32_t SWEEP_GROUP = 2, SWEEP_TILE = 8192;
constexpr uint32_t SWEEP_THREADS[SWEEP_KERNELS] = {128, 64, 128, 64, 128, 512, 256};   // most threads of a CTA
constexpr uint32_t SWEEP_ONE_THREADS = 512;   // with one CTA an SM

// Sections of an expression: their values take 512 bytes (FP8 576) of shared
// memory each.  (With at most 32, one warp folded all 512 sources of {64, 8}.)
constexpr uint32_t SWEEP_TEAM_MAX = 128;
constexpr uint32_t SWEEP_TEAM_STATIC = 32;   // whose values lie in static shared memory
// In a fold pass of few units every warp folds one source after the other,
// about 300 cycles each, while most of an SM idles: below eight units an SM
// the sections go to the warps of a CTA, as many as fill the SMs
// (SWEEP_TEAM_WARPS in all).  Measured without / with, All-reduce of 64 ranks
// x 64 KiB 12.7 / 9.4 us, Reduce of 64 ranks x 16 KiB 10.8 / 6.1 us; at 1024
// units (16 ranks x 512 KiB) 7.3 / 5.2 us, at 2048 (1 MiB) 8.6 / 10.6 us.
constexpr uint32_t SWEEP_TEAM_UNITS = SWEEP_SMS * 8, SWEEP_TEAM_WARPS = SWEEP_SMS * 32;
// More than 32 sections: every warp evaluates the expression of all their values,
// so the lines lie earlier.  Reduce, F32, by one warp / by 64 sections of {64, 8}
// (us): 2 units 67 / 14, 128 units 67 / 16, 512 76 / 39; 128 of {128, 8}: 132 / 25,
// 133 / 29, 146 / 73, 1024 units 148 / 164; 50 of {50, 2}, BF16: 512 units 26.8 / 29.3.
// Where a level has fewer sections, by 2 or 64 of {2, 32, 4}: 1 unit 32 / 12, 128
// 32 / 14; by 4 or 64 of {4, 16, 4}: 512 units 22 / 23.  FP8 values take as long to
// fold as sources, so there fewer stay better: {4, 16, 4}, 128 units, 22.5 / 27.7.
constexpr uint32_t SWEEP_TEAM_MANY = SWEEP_SMS * 3, SWEEP_TEAM_FEW = SWEEP_SMS * 2;

// token of one source, in evaluation order: START the accumulator with it
// (first saving the old one when PUSH is set), else combine it; then up to
// 12 two-bit operations from bit 8 on, the first in the low bits (every
// operator gives the same bits for both orders of two values, so the kernels
// take POP and JOIN alike)
constexpr uint32_t TOK_START = 1u, TOK_PUSH = 2u, TOK_OPS = 8u;
enum : uint32_t {
  TOK_ROUND = 1,   // round the accumulator to the payload
  TOK_POP = 2,     // accumulator = combine(saved value, accumulator)
  TOK_JOIN = 3     // accumulator = combine(accumulator, saved value)
};

struct SweepClass {
  unsigned long long nbytes;   // bytes of every operand of a member
  unsigned long long ptr;      // first operand pointer of member 0 (members at a stride of nsrc + ndst)
  uint32_t unit0;              // first unit of the class within its launch
  uint32_t upm;                // units per member
  uint32_t nmem;
  uint32_t nsrc, ndst;
  uint32_t tok;                // first of the nsrc tokens
  uint32_t meta;               // sweep_meta
  uint32_t group;              // destinations that one unit stores (copies; folds store all)
  // an expression in two steps (team > 1): `team` sections of consecutive
  // sources, evaluated apart, then an expression of their values.  From token
  // ttok: the sections' nsrc tokens, their team + 1 bounds, team tokens.
  uint32_t team;
  uint32_t ttok;
  uint32_t pad[2];
};
static_assert(sizeof(SweepClass) == 64, "class layout");
// dtype (4 bits) | operator (3) | log2 of the access width (3) | vectors per lane (5) | kernel (3)
HICCL_HD inline uint32_t sweep_meta(uint32_t dt, uint32_t rop, uint32_t lw, uint32_t v, uint32_t kern) {
  return dt | (rop << 4) | (lw << 7) | (v << 10) | (kern << 15);
}
HICCL_HD inline uint32_t sweep_dtype(uint32_t m) { return m & 15u; }
HICCL_HD inline uint32_t sweep_rop(uint32_t m) { return (m >> 4) & 7u; }
HICCL_HD inline uint32_t sweep_lw(uint32_t m) { return (m >> 7) & 7u; }
HICCL_HD inline uint32_t sweep_v(uint32_t m) { return (m >> 10) & 31u; }
HICCL_HD inline uint32_t sweep_kernel(uint32_t m) { return (m >> 15) & 7u; }

// A launch of more than SWEEP_PREFIX classes finds a unit's class from hints:
// hint i is the class (within the launch) of unit i << SWEEP_HINT_SHIFT, so
// the class lies between two of them.  (By a binary search over the classes in
// memory, eight dependent loads a warp, the group of 256 collectives of 4 KiB to
// 16 MiB took 2.21 ms instead of 1.92.)
constexpr uint32_t SWEEP_HINT_SHIFT = 7;
struct SweepLaunch {
  uint32_t kernel;
  uint32_t class_lo, class_hi;
  uint32_t units;
  uint32_t threads;
  uint32_t stack_words;        // 32-bit words of saved values per thread
  uint32_t hint;               // first hint
  uint32_t sections;           // of the class that has most (launches of teams)
};

// ---------------------------------------------------------------------------
// host-side plan
// ---------------------------------------------------------------------------

// The sweep of a plan (hiccl_sweep.cpp); valid is false where the program
// does not reduce to independent expressions.
struct Sweep {
  bool valid = false;
  std::vector<SweepClass> classes;            // grouped by launch
  std::vector<uint32_t> toks, hints;
  std::vector<unsigned long long> ptrs;
  std::vector<SweepLaunch> launches;
  uint32_t depth = 0;                         // saved values of the deepest expression
};

// bytes of its tables on the device
inline size_t sweep_bytes(const Sweep &w) {
  return std::max<size_t>(w.classes.size() * sizeof(SweepClass) + w.ptrs.size() * 8 + (w.toks.size() + w.hints.size()) * 4, 16);
}
constexpr size_t TRACE_BYTES = 6 * sizeof(unsigned long long);   // of a work item

struct Loc {
  unsigned long long addr;   // device address, or relay-arena offset when scratch
  int32_t rank;
  uint8_t scratch;
};

struct HStep {
  uint8_t kind;            // OP_COPY / OP_REDUCE
  int8_t level;            // hierarchy level crossed; -1 local
  int32_t prim;
  int32_t epoch;
  int32_t branch;
  int32_t channel;
  unsigned long long nbytes;
  uint32_t loc0;           // first Loc: nsrc sources then ndst destinations
  uint32_t nsrc;
  uint32_t ndst;
  unsigned long long slot;
  uint32_t local;          // emission index inside its piece (same tree position in every channel)
  uint32_t dtype;          // payload type of the step's communicator
  uint32_t rop;            // reduction operator (hiccl_op_t) of a reduce
  uint32_t pad3;
};

struct Prim {
  int kind;                                // 0 multicast, 1 reduction
  int op = 0;                              // hiccl_op_t of a reduction
  int root;
  std::vector<int> leaves;                 // sorted, distinct
  size_t count;
  std::vector<unsigned long long> send;    // per rank (0 = none)
  std::vector<unsigned long long> recv;
  int epoch;
};

// A range that a primitive reads or writes, and those of a program: primitive
// i has all[of[i]] .. all[of[i + 1] - 1], its reads first.
struct Range {
  unsigned long long lo, hi;
  int prim;
  bool write;
  int rank = -1;   // owner of the buffer
};
struct Ranges {
  std::vector<Range> all;
  std::vector<size_t> of;
};

// Byte ranges of two primitives that overlap across a fence, one of them written.
struct Conflict {
  uint32_t later, earlier;   // primitives
  bool same;                 // the ranges are equal
  bool rewrites;             // both write
};

struct DevState;   // defined by the runtime

struct Plan {
  std::vector<int> hierarchy;
  int stripe = 1, pipeline = 1;
  unsigned long long seg = SEG_BYTES;      // segment bytes (seg_bytes_of(dtype))
  std::vector<HStep> steps;                // in execution (slot) order
  std::vector<Loc> locs;
  std::vector<uint32_t> pred_off, preds;   // CSR of predecessors (by new index)
  std::vector<uint32_t> succ_off, succ;    // CSR of successors
  std::vector<DevEntry> entries;
  std::vector<uint32_t> item_off;
  std::vector<DevRun> runs;
  std::vector<uint32_t> run_off;
  std::vector<uint32_t> nent;             // entries covering each step
  unsigned long long scratch_bytes = 0;
  std::vector<unsigned long long> level_bytes;
  unsigned long long hbm_read = 0, hbm_write = 0;
  unsigned long long stages = 0, slots = 0;
  Sweep sweep;
  bool valid = false;
  bool corrupted = false;                  // by hiccl_debug_corrupt: never runs
};

// Host image of the executor's read-only arrays for a plan whose relay
// offsets resolve against relay_base (hiccl_plan.cpp, build_image).
struct TableImage {
  std::vector<unsigned long long> ptrs;   // every location, resolved
  std::vector<uint32_t> indeg;            // per step
  std::vector<unsigned char> recs;        // work-item records
  std::vector<DevItem> items;             // per work item
};
void build_image(const Plan &p, unsigned long long relay_base, TableImage &im);
// bytes of TableImage::recs for plan p, without building the image
unsigned long long record_bytes(const Plan &p);

}  // namespace hiccl

struct hiccl_comm {
  int P = 0;
  hiccl_dtype_t dtype = HICCL_F32;
  int esize = 4;
  int epochs = 1;
  std::vector<hiccl::Prim> prims;
  enum State { COMPOSING, PLANNED, READY, RUNNING } state = COMPOSING;
  bool group = false;   // built by hiccl_group from other communicators' plans
  // options
  unsigned long long timeout_ns = 1000000000ull;
  int ctas_per_sm = 2;
  int threads = 256;
  unsigned long long item_bytes = 49152;   // set per payload at creation
  int order = 1;
  unsigned long long slot_items = 0;   // 0: whole rounds over the executor grid
  int trace = 0;
  int ring = 1;                       // ring(n) of Sec. 4.4; 1 = tree only
  hiccl::Plan plan;
  hiccl::DevState *dev = nullptr;
  std::string err;
};

namespace hiccl {
hiccl_status_t fail(hiccl_comm *c, hiccl_status_t st, const std::string &msg);
// Run the body of a C-ABI call so that no C++ exception leaves it: host
// memory exhaustion becomes HICCL_ERR_NOMEM, anything else HICCL_ERR_INVALID,
// with the message on `c` where there is one.
template <typename F>
hiccl_status_t guarded(hiccl_comm *c, F &&body) noexcept {
  hiccl_status_t st;
  const char *msg;
  try {
    return body();
  } catch (const std::bad_alloc &) {
    st = HICCL_ERR_NOMEM;
    msg = "out of host memory";
  } catch (...) {
    st = HICCL_ERR_INVALID;
    msg = "internal error";
  }
  try {
    return fail(c, st, msg);
  } catch (...) {
    return st;
  }
}
// the sweep of c's program over `hierarchy` (ring_lvl: level of the ring's
// nodes; conflicts across fences ordered by the later primitive), and the
// union of several (hiccl_sweep.cpp)
void build_sweep(const hiccl_comm &c, const std::vector<int> &hierarchy, int ring_lvl,
                 const Ranges &ranges, const std::vector<Conflict> &conflicts, Sweep &sw);
void group_sweep(const std::vector<const Sweep *> &members, Sweep &sw);
// Consistency of a sweep before it reaches the GPU (ranges: of c's program,
// empty for a group); false with the first violation in `why`.
bool check_sweep(const hiccl_comm &c, const Ranges &ranges, const Sweep &sw, std::string &why);
// factorize c's program again (hiccl_plan.cpp), keeping c's state
hiccl_status_t replan(hiccl_comm *c, const std::vector<int> &hierarchy, int stripe, int pipeline);
// runtime entry points (hiccl_runtime.cu)
hiccl_status_t dev_upload(hiccl_comm *c);
void dev_release(hiccl_comm *c);
// after a change of CTAS_PER_SM
hiccl_status_t dev_options(hiccl_comm *c);
// CTAs of an executor launch of c on the calling thread's current device
// (SMs x resident CTAs per SM for c's THREADS and CTAS_PER_SM); 0 when no
// device can be queried
unsigned long long exec_grid(const hiccl_comm &c);
}  // namespace hiccl
