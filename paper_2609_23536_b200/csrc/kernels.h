// Kernel parameter blocks and host-side launch descriptors shared by the execution layer.
// Every kernel of the library takes exactly one by-value parameter struct, so that a launch is fully
// described by (function, grid, block, dynamic shared memory, parameter bytes) and the same description
// serves an eager launch, a CUDA-graph kernel node and a later in-place update of that node.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <utility>
#include <vector>

namespace qe {

// ---- device-resident layer state (lives at the start of the caller's workspace) -------------------------------
struct DevState {
  float scale[4];              // indexed by qe_tensor_class
  float scale_inv[4];
  uint32_t count[4];           // commits so far
  uint32_t pending_amax[4];    // non-negative FP32 bit patterns, accumulated with atomicMax, cleared by commit
  unsigned long long token;    // effect token as counted on the device
  float cache_sinv_W;          // inverse weight scale at the last cache refresh
  uint32_t status;             // error bits ORed in by kernels whose bounded waits expired
  float slot_sinv_X[64];       // inverse scales snapshotted when X_m / dY_m were quantised (per tape slot)
  float slot_sinv_G[64];
  uint32_t ticket;             // "last CTA" counter of the kernel whose tail performs the commit; self-resetting
  uint32_t wmax[4];            // bit pattern of max(history ring) per class, kept by the commit (derived state)
  uint32_t status_all;         // scratch of the multi-layer boundary: OR of several layers' status words
  uint32_t commits;            // whole-step calls whose first layer this is: Announce::word
  uint32_t rows_done[32];      // launches of chained GEMMs: parts of 256 rows of this layer's result that are stored; 0 between them
  uint32_t pad[5];             // header is 768 bytes; history rings [4][H] follow
};
static_assert(sizeof(DevState) == 768, "DevState layout");

struct CommitParams {
  DevState* st;                // null: nothing to commit
  float* hist;                 // [4][H]
  uint32_t H;
  uint32_t class_mask;         // bit c set: commit class c from pending_amax[c] (or from amax_override)
  float pow2_neg_margin;       // 2^-margin
  uint32_t early_mask;         // GEMM launches: classes whose amax is complete when the launch starts (committed then, with
                               // the token); class_mask holds the ones its own epilogue completes
  uint32_t bump_token;         // 1 for F and dI, 0 otherwise
  uint32_t pad;
  const float* amax_override;  // if non-null: value to push for the single class in class_mask
};

struct QuantParams {
  const uint16_t* x;           // bf16 [rows, cols]
  uint8_t* q;                  // fp8 [rows, cols]
  uint8_t* qT;                 // fp8 [cols, rows] or null (a launch of its own only)
  uint32_t rows, cols;
  const float* scale;          // device scalar read by every thread
  const float* sinv_src;       // if non-null, block 0 copies *sinv_src to *sinv_dst (tape snapshot)
  float* sinv_dst;
  uint32_t* amax_bits;         // atomicMax target or null
  int32_t fmt;                 // 0 = E4M3, 1 = E5M2
  uint32_t pad;
  CommitParams commit;         // performed by the last block to finish (commit.st != null)
};


// A launch of casts that need not wait for the GEMM launch before it, which is only to have made its early commits (it counts
// the problems that have, in *word; announce_commits).  Null: the casts wait.
struct Announce {
  uint32_t* word = nullptr;
  uint32_t count = 0;          // what *word has come to by then
};

constexpr uint32_t kMaxCasts = 128;  // of one launch
template <int N>
struct QuantMultiParams {
  QuantParams q[N];
  uint32_t block_end[N];       // cumulative block counts
  uint32_t n;
  uint32_t commits_count;      // Announce
  const uint32_t* commits;
};

struct AmaxParams {
  const uint4* x;              // bf16, 8 per vector
  uint64_t nvec;
  float* partials;
  float* out;
  uint32_t nparts;
  uint32_t pad;
};

struct AccumParams {
  float4* dst;
  const float4* src;
  uint64_t nvec;
  int32_t accumulate;
  int32_t pad;
};

// Sum of M bf16 views (view m at views + m * view_vec 16-byte vectors) into FP32, added in view order.
struct ArenaReduceParams {
  const uint4* views;   // 8 bf16 per vector
  float4* dst;          // 2 vectors of 4 FP32 per input vector
  uint64_t view_vec;    // vectors per view (= N*K / 8)
  uint32_t M;
  uint32_t pad;
};

// Tile widths the GEMM can be run with: the B operand's TMA box has half as many rows (each CTA of a pair loads half).
constexpr uint32_t kNumTileWidths = 3;
constexpr uint32_t kTileWidths[kNumTileWidths] = {256, 128, 64};
// K blocks of 128 that a box of an operand holds: one where tiles are 256 columns wide, else two; an operand in the A role has
// a map for either.
constexpr uint32_t blocks_of(uint32_t width) { return width ? 2u : 1u; }
constexpr uint32_t a_map_of(uint32_t width) { return width ? 1u : 0u; }

constexpr uint32_t kMaxSegments = 8;

// D = (A . B^T) * (*alpha_a * *alpha_b), or the sum of several such products over tensors of the same shape at equal distances
// (the tape slots of a layer): an operand's map spans all of them.
struct GemmParams {
  CUtensorMap tmA;             // A: boxes of 128 rows x 128 contraction bytes x blocks_of(width), 128-byte swizzle
  CUtensorMap tmB;             // B: tile_n / 2 rows, likewise (MN-major: swizzled over tile_n / 2 bytes)
  CUtensorMap tmD;             // D [M, N] (bf16, FP32 or FP8 bytes), box 32 x 32 (sum: 128 x 32), for the epilogue's bulk stores
  const float* alpha_a;        // [slot]
  const float* alpha_b;
  uint8_t slot_a[kMaxSegments], slot_b[kMaxSegments];  // of each product
  uint32_t M, N, Kc;
  uint32_t tile_n;             // columns per tile
  uint32_t nseg;               // products; more than one: an FP32 output (epi 1, 2) that receives them one after the other, as
                               // nseg launches would have added them
  uint32_t idesc;              // tcgen05 instruction descriptor (formats, majors, shape)
  uint32_t b_desc_hi, b_step;  // B's shared-memory descriptor: high word; address advance (16-byte units) per 32 contraction elements
  uint8_t a_mn, b_mn;          // operand given MN-major (as [Kc, M] / [Kc, N] bytes)
  uint8_t sum, pad;            // FP32 result of one product or several that gemm_fp8_pair_wide_kernel keeps in registers: after all
                               // other problems of the launch; tmD's box has 128 rows
  uint32_t ldo;
  void* out;                   // bf16 or FP32 [M, N], row pitch ldo elements
  uint32_t* amax_bits;         // or null
  // epi 3: the bf16-rounded result is not stored; it is quantised for the consuming linear as that linear's own
  // cast kernel would have done: q = fp8(fp32(bf16(D)) * *out_scale), max|bf16(D)| also into *amax_bits2, and
  // *sinv_dst = *sinv_src (the consumer's tape snapshot)
  const float* out_scale;
  int32_t out_fmt;             // 0 = E4M3, 1 = E5M2
  int32_t epi;                 // 0 bf16 (+amax), 1 FP32 overwrite, 2 FP32 accumulate, 3 FP8 hand-off (above)
  uint32_t* amax_bits2;        // or null
  const float* sinv_src;
  float* sinv_dst;
  uint32_t* status;
  CommitParams commit;         // performed by the last CTA to finish (commit.st != null)
};

// One GEMM as the launch builders take it: everything the kernel needs except what follows from the tile width (tmA, tmB,
// tile_n, idesc, b_desc_hi, b_step), which is filled from the fields below.
struct GemmDesc : GemmParams {
  uint32_t a_fmt, b_fmt;       // 0 = E4M3, 1 = E5M2
  const CUtensorMap* mapA;     // [2]: a_map_of(width); the launch reads those of the width it chooses (gemm_width)
  const CUtensorMap* mapB;     // [kNumTileWidths]
  CommitParams before{};       // of a launch of its own: GemmLaunchParams::before
  bool chained = false;        // make_gemm_group: each problem's A is the result of the one before (FP8 hand-off)
  GemmDesc() : GemmParams{}, a_fmt(0), b_fmt(0), mapA(nullptr), mapB(nullptr) { nseg = 1; }
  void operands(const CUtensorMap* a, const float* alphas_a, uint32_t slot_of_a, const CUtensorMap* b, const float* alphas_b, uint32_t slot_of_b) {
    mapA = a, mapB = b, alpha_a = alphas_a, alpha_b = alphas_b;
    slot_a[0] = (uint8_t)slot_of_a, slot_b[0] = (uint8_t)slot_of_b;
  }
  void add_product(uint32_t slot_of_a, uint32_t slot_of_b) {
    slot_a[nseg] = (uint8_t)slot_of_a, slot_b[nseg] = (uint8_t)slot_of_b;
    ++nseg;
  }
};

// Independent GEMMs computed by one launch: tiles are numbered problem after problem.
template <int NP>
struct GemmLaunchParams {
  uint32_t* commits;           // Announce: the next kernel in the stream may start before this one ends and reads what the early
  uint32_t commits_op;         // part commits.  1: a problem is counted after that and the next kernel let go; 2: set to zero
  uint32_t n;
  uint32_t tile_end[NP];       // cumulative tile counts
  uint32_t* ticket;            // counts the CTAs that are done, where a problem has a commit in the tail; else null
  CommitParams before;         // launches of one problem: a class whose amax the launch before completed (before.st != null)
  GemmParams prob[NP];
};
constexpr uint32_t kLaunchChained = 4, kMaxChained = 16;  // problems of a launch of chained GEMMs, at least and at most
constexpr uint32_t kMaxProblems = 56;  // of a launch: what a kernel's parameter space of 32764 bytes holds
// ... and of one whose problems commit scales at its start, a CTA each: the grid has that many at least
inline uint32_t most_committing(int num_sms) {
  const uint32_t ctas = num_sms < 4 ? 2u : (uint32_t)num_sms / 2u * 2u;
  return ctas < kMaxProblems ? ctas : kMaxProblems;
}

// ORs the status words of up to 64 layers into *out (first chunk: out = OR; later chunks: out |= OR).
struct StatusGatherParams {
  const uint32_t* src[64];
  uint32_t* out;
  uint32_t n;
  uint32_t accumulate;
};

// Bytes of a parameter block.  Those of a launch of one problem live inside the object: the standalone calls, and with
// them the one that promises to touch no allocator, take no heap memory.
class ParamBytes {
 public:
  static constexpr size_t kInline = 768;
  ParamBytes() = default;
  ParamBytes(const ParamBytes& o) { *this = o; }
  ParamBytes(ParamBytes&& o) noexcept { *this = std::move(o); }
  ParamBytes& operator=(const ParamBytes& o) {
    if (this == &o) return *this;
    if (o.n_ > kInline) more_.assign(o.more_.begin(), o.more_.end());
    else __builtin_memcpy(here_, o.here_, o.n_);
    n_ = o.n_;
    return *this;
  }
  ParamBytes& operator=(ParamBytes&& o) noexcept {
    if (this == &o) return *this;
    if (o.n_ > kInline) more_ = std::move(o.more_);
    else __builtin_memcpy(here_, o.here_, o.n_);
    n_ = o.n_;
    o.n_ = 0;
    return *this;
  }
  void resize(size_t n) {  // all bytes zero
    if (n > kInline) more_.assign(n, 0);
    else __builtin_memset(here_, 0, n);
    n_ = n;
  }
  size_t size() const { return n_; }
  unsigned char* data() { return n_ > kInline ? more_.data() : here_; }
  const unsigned char* data() const { return n_ > kInline ? more_.data() : here_; }

 private:
  size_t n_ = 0;
  alignas(64) unsigned char here_[kInline];
  std::vector<unsigned char> more_;
};

// One launch, self-contained.
struct Launch {
  const void* func = nullptr;
  dim3 grid{1, 1, 1}, block{1, 1, 1};
  uint32_t smem = 0;
  bool cooperative = false;  // its blocks wait on one another
  ParamBytes params;    // the parameter block, without an unused tail ...
  uint32_t nbytes = 0;  // ... of a block of this size
  template <class P>
  void set(const P& p) {
    params.resize(sizeof(P));
    __builtin_memcpy(params.data(), &p, sizeof(P));
    nbytes = sizeof(P);
  }
  // The whole block as the runtime wants it (valid as long as the launch and the buffer are).
  struct Block { alignas(64) unsigned char bytes[32768]; };
  void* args_block(Block* tmp) const {
    if (params.size() == nbytes) return const_cast<unsigned char*>(params.data());
    __builtin_memcpy(tmp->bytes, params.data(), params.size());
    return tmp->bytes;
  }
};

Launch make_quantize(const QuantParams& p);
Launch make_quantize_multi(const QuantParams* casts, uint32_t n, const Announce& early = {});  // 1..kMaxCasts independent casts without transposed copies in one launch
Launch make_commit(const CommitParams& p);
Launch make_status_gather(const StatusGatherParams& p);
Launch make_amax_pass1(const AmaxParams& p);
Launch make_amax_pass2(const AmaxParams& p);
Launch make_accumulate(const AccumParams& p);
Launch make_arena_reduce(const ArenaReduceParams& p);
Launch make_gemm(const GemmDesc& p, int num_sms);
// One launch for n = 2..kMaxProblems GEMMs (each may carry its own commit tail); false if there are more, or if they are chained and
// better launched one by one.
// (most_committing, where they commit scales at the launch's start)
bool make_gemm_group(const GemmDesc* probs, uint32_t n, int num_sms, Launch* out);
// Whether the device, as the stream may use it, holds all blocks of a launch of chained GEMMs at once.  (A device whose units have odd
// numbers of SMs, or a part of one, may not; launches one by one run on any number.)
bool chained_fit(int num_sms, cudaStream_t stream);
uint32_t announce_commits(Launch* gemm, uint32_t* word);  // the launch is to count its problems in *word; how many that are
void withdraw_commits(Launch* gemm, uint32_t* word);      // the launch is to set *word to zero
uint32_t gemm_width(const GemmDesc* probs, uint32_t n, int num_sms);  // index of the tile width the launch of these will have
cudaError_t gemm_prepare();  // opt in to the dynamic shared memory the GEMM needs (once per device)
// Whether M fills whole 256-row tiles.  The kernels take any multiple of 128, and the layers' MN-major operands come with any;
// shared launches, the hand-off (of N) and MN-major operands of the standalone calls are offered for whole tiles only.
bool whole_row_tiles(uint32_t M);
constexpr uint32_t kAmaxPartials = 2048;

}  // namespace qe
