// The contraction of k_umma.cu (see there for the matrix product and the operand images) for
// the FP32 tier, on pairs of CTAs: FP16 hi + lo operands, and accumulation groups of one or two
// chunks, so that the accumulator's rounding toward zero stays below the phasors' own error.
//
// A pair's MMA (tcgen05.mma.cta_group::2, M = 256, N = 2 NT rounded up to a multiple of 32)
// takes two row tiles at once: each
// CTA holds its own 128 rows of A and one half of B (rank 0 the re-rows, rank 1 the im-rows),
// so that a chunk's B crosses L2 once per pair.  Per CTA, warp-specialised:
//   warps 0-7    produce A for the CTA's 128-row tile in shared memory (one row per thread, 16
//                pixels of each stage);
//   warps 8-15   add each finished accumulation group into FP32 sums held in registers and
//                write a unit's sums once at its end.  Two accumulators in tensor memory
//                alternate, so this runs beside the next group's MMAs and short groups (the
//                accumulator rounds toward zero) cost little;
//   warp 16      allocates tensor memory; one thread of the leader (rank 0) issues the MMAs,
//                one of the peer tells the leader when its part of a stage is there;
//   warp 17      decodes the pair's work units and bulk-copies the phases of the tile's channels;
//   warp 18      bulk-copies the CTA's half of each chunk's B images.
// setmaxnreg moves registers from the other warps to the summing ones.  Every wait is bounded
// in time and a timeout sets a status bit instead of hanging.
// Measured on a frame of 256 x 256 pixels (V = 12, N_s = 256, L = 128), kernel alone: 240 us in
// groups of two chunks and 232 in groups of 40, where one CTA per tile with A in tensor memory
// and the accumulator drained by the producers took 229-235 us in groups of 40 and 407-409 in
// groups of 4; the CUDA cores took 2790.  Bound by the MMAs (348,000 of about 420,000 cycles;
// the SM clock falls to 1.75-1.9 GHz under them) and by shared memory, whose port the operands'
// writes and the MMAs' reads fill to about 80%.
#include <algorithm>

#include "rsim_internal.h"
#include "umma.h"

namespace rsim {
namespace {

using namespace umma;

constexpr int kPixStages = 3;              // ring of staged pixel phases
constexpr int kPixChunks = 4;              // chunks per slot of that ring
constexpr int kUnitSlots = 4;              // ring of work units
constexpr int kMaxCh = 8;                  // channels a row tile may span for staging
constexpr int kAWarps = 8;                 // A producers, two per lane quarter
constexpr int kAPx = kChunkPx / (kAWarps / 4);  // pixels per A warp per stage
constexpr int kSumWarps = 8;               // running sums in registers, two per lane quarter
constexpr int kMmaWarp = kAWarps + kSumWarps;  // then the pixel loader, the B loader, an idle warp
constexpr int kThreads = 32 * (kMmaWarp + 4);  // whole warpgroups: 2 of producers, 2 of sums, 1 of the rest
// Registers a thread of each warpgroup (setmaxnreg): 256 x 64 + 256 x 152 + 128 x 48 =
// 61,440, what a launch of 640 threads at 96 registers holds.
constexpr int kRegsLaunch = 96, kRegsA = 64, kRegsSum = 152, kRegsRest = 48;
static_assert(32 * (kAWarps * kRegsA + kSumWarps * kRegsSum + 4 * kRegsRest) <= kThreads * kRegsLaunch,
              "the warpgroups' registers fit the launch's");
constexpr uint32_t kFineLong = 20000 / kChunkPx;  // chunks of a frame from which groups are long
// The accumulator rounds toward zero, so a group's sum comes out short by about half a unit in
// the last place of each addition at its size: by 0.8 x 2^-23 of itself in groups of one chunk
// (four additions of A_hi B_hi at a quarter to all of the size) and by 2.4 x 2^-23 in groups of
// two (twelve more).  Measured against the CUDA-core sum, which has the same phasors, over 128 to
// 262,144 pixels and equal, log-normal and 1/R^2 strengths of one and of random phase: 0.9 to
// 1.0e-7 and 2.6 to 2.9e-7.  A unit's sums are lengthened by it.  Error with strengths of one
// phase (rendered scenes; the CUDA-core sum's in brackets) without and with it: 2,048 pixels
// 2.5 -> 1.9e-7 (2.5e-7), 40,000 4.2 -> 1.8e-7 (1.7e-7), 262,144 4.1 -> 1.7e-7 (1.9e-7); of
// random phase 3.2 -> 2.6e-7 (4.1e-7), 5.2 -> 3.4e-7 (5.8e-7) and 5.6 -> 3.8e-7 (1.4e-6).
constexpr float kShort1 = 0.8f * 0x1p-23f, kShort2 = 2.4f * 0x1p-23f;
constexpr int kPartBytes = 128 * 128;      // one 16-bit part of a stage's A (128 rows) or of its half of B
constexpr int kAccCols = 256;              // columns of one accumulator (N <= 256 FP32)
constexpr int kTmemCols = 512;             // two accumulators
constexpr int kStages = 3;                 // operand stages in shared memory: A hi, A lo, B hi, B lo
constexpr int kStageBytes = 4 * kPartBytes;

// Fast-time/channel phases of kPixChunks chunks, staged by the pixel loader (bulk copies).
struct PixStage {
  uint32_t a[kMaxCh][kPixChunks * kChunkPx];  // fast-time increments of the tile's channels
  uint32_t c[kMaxCh][kPixChunks * kChunkPx];  // spatial phases of the tile's channels
};

// A work unit, decoded once by the pixel loader: a row tile, a column tile and a range of
// the frame's 32-pixel chunks.
struct Unit {
  int f, mt, nt, s;   // frame (-1: no more work), row tile, column tile, pixel split
  uint32_t c0, c1;    // chunks c0 .. c1 - 1 (a frame has at most 2^26)
  int group;          // chunks per accumulation group, at most
  int v_first, span;  // the channels its rows lie in
};

struct Shared {
  Unit unit[kUnitSlots];
  uint64_t full[kStages];    // the stage's A and half of B are here; the leader's waits for the
                                // peer's word too, which one thread of the peer passes on
  uint64_t empty[kStages];   // the MMAs are done with the stage
  uint64_t pix_full[kPixStages];
  uint64_t pix_empty[kPixStages];
  uint64_t unit_full[kUnitSlots];
  uint64_t unit_empty[kUnitSlots];
  uint64_t acc_full[2];   // a group is summed in the accumulator
  uint64_t acc_empty[2];  // leader: both CTAs have read it out
  uint64_t fin;
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, Shared* sh, unsigned* status) {
  return umma::mbar_wait(b, parity, &sh->abort, status);
}
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, Shared* sh, unsigned* status) {
  return umma::warp_wait(b, parity, &sh->abort, status);
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Instruction descriptor of kind::f16: FP16 operands, FP32 accumulator, K-major A and B, M = 256 (the
// pair).
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// All MMAs of one 32-pixel operand stage (K = 64 16-bit elements = four K = 16 steps).  `a`,
// `b`: descriptors of the stage's hi A and hi B (the lo parts lie kPartBytes on); a K step
// moves both by 32 bytes (2 in the descriptor's 16-byte address field).  `acc` = 0 starts a
// new accumulation with the stage's first MMA.  The small products come first, so that in a new
// accumulation only the four A_hi B_hi are added to (and rounded toward zero at) the sum's full
// size.
#define RSIM_MMA(a, b, en) "tcgen05.mma.cta_group::2.kind::f16 [%0], " a ", " b ", %3, " en ";\n\t"
#define RSIM_STEP(x, from, n) "add.s64 " x ", " from ", " n ";\n\t"
__device__ __forceinline__ void mma_stage(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, t;\n\t.reg .b64 x, y, u, v;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 t, %3, 0;\n\t"
      RSIM_STEP("u", "%1", "%5") RSIM_STEP("v", "%2", "%5")
      RSIM_MMA("%1", "v", "p") RSIM_MMA("u", "%2", "t")
      RSIM_STEP("x", "%1", "2") RSIM_STEP("y", "%2", "2") RSIM_STEP("u", "u", "2") RSIM_STEP("v", "v", "2")
      RSIM_MMA("x", "v", "t") RSIM_MMA("u", "y", "t")
      RSIM_STEP("x", "x", "2") RSIM_STEP("y", "y", "2") RSIM_STEP("u", "u", "2") RSIM_STEP("v", "v", "2")
      RSIM_MMA("x", "v", "t") RSIM_MMA("u", "y", "t")
      RSIM_STEP("x", "x", "2") RSIM_STEP("y", "y", "2") RSIM_STEP("u", "u", "2") RSIM_STEP("v", "v", "2")
      RSIM_MMA("x", "v", "t") RSIM_MMA("u", "y", "t")
      RSIM_MMA("x", "y", "t")
      RSIM_STEP("x", "x", "-2") RSIM_STEP("y", "y", "-2") RSIM_MMA("x", "y", "t")
      RSIM_STEP("x", "x", "-2") RSIM_STEP("y", "y", "-2") RSIM_MMA("x", "y", "t")
      RSIM_MMA("%1", "%2", "t") "}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc), "n"(kPartBytes >> 4)
      : "memory");
}
#undef RSIM_MMA
#undef RSIM_STEP

// Completes one arrival on the barrier at `b`'s place in each CTA of the pair once the MMAs
// issued so far are done (`peer`: its address in the peer's shared memory).
__device__ __forceinline__ uint32_t peer_addr(const void* p) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 1;" : "=r"(a) : "r"(smem_u32(p)));
  return a;
}
__device__ __forceinline__ void mma_commit(uint64_t* b) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%1];" ::"r"(smem_u32(b)),
      "r"(peer_addr(b))
      : "memory");
}

struct Geo {
  int mpairs, ntiles, NT, splits, upf, direct, F;
  int NH;                // accumulator columns of one half (re or im): NT, rounded up to 16
  int total_units;       // work units (frame, pair of row tiles, column tile, split)
  int64_t sstride;       // complex elements of one split's tiled partial sums
  const int32_t* order;  // frames by decreasing valid-pixel count
};

// Unit u as the CTA of rank `rank` in its pair sees it.
__device__ __forceinline__ Unit decode(const Geo& g, const FrameIO* frames, const Consts& k, int u, int rank) {
  Unit x;
  const int fi = u / g.upf;
  x.f = g.order ? g.order[fi] : fi;
  // row tile fastest: the CTAs running at the same time share a pixel range and so the
  // same slow-time operand images in L2
  int r = u % g.upf;
  x.mt = 2 * (r % g.mpairs) + rank;
  r /= g.mpairs;
  x.nt = r % g.ntiles;
  x.s = r / g.ntiles;
  const uint32_t nch = (uint32_t)((frames[x.f].meta[0] + kChunkPx - 1) / kChunkPx);
  // one chunk a group (error 2.6 to 3.0e-7 with equal strengths), two for long sums (3.0 to
  // 3.8e-7; in groups of one the frame of 46,000 valid pixels takes 327 us instead of 275)
  x.group = nch < kFineLong ? 1 : 2;
  x.c0 = nch * (uint32_t)x.s / (uint32_t)g.splits;
  x.c1 = nch * (uint32_t)(x.s + 1) / (uint32_t)g.splits;
  const int64_t rows = (int64_t)k.V * k.Ns;
  const int64_t r0 = (int64_t)x.mt * 128;
  const int64_t r1 = (r0 + 127 < rows ? r0 + 127 : rows - 1);
  x.v_first = (int)(r0 / k.Ns);
  x.span = (r0 < rows) ? (int)(r1 / k.Ns) - x.v_first + 1 : 0;
  return x;
}

// Accumulation groups of a unit: its chunks c0 .. c1 - 1 cut into the fewest equal groups
// of at most `gmax` chunks, one drain each (a unit without chunks still has one group,
// whose drain writes zeros).  Equal groups spend no drain on a short tail group.
__device__ __forceinline__ uint32_t unit_groups(uint32_t chunks, int gmax) {
  return chunks > 0 ? (chunks + gmax - 1) / gmax : 1;
}
// Chunks of group k: the first chunks mod ngr groups hold one more than the others.
__device__ __forceinline__ uint32_t group_chunks_of(uint32_t chunks, uint32_t ngr, uint32_t k) {
  return chunks / ngr + (k < chunks % ngr ? 1 : 0);
}

// Next work unit from the ring filled by the pixel loader; false when there is none.
__device__ __forceinline__ bool next_unit(Shared* sh, uint32_t ui, unsigned* status, Unit* u, bool warp_collective) {
  const uint32_t slot = ui % kUnitSlots, ph = (ui / kUnitSlots) & 1u;
  const bool ok = warp_collective ? warp_wait(&sh->unit_full[slot], ph, sh, status)
                                  : mbar_wait(&sh->unit_full[slot], ph, sh, status);
  if (!ok) return false;
  *u = sh->unit[slot];
  if (warp_collective) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&sh->unit_empty[slot]);
  } else {
    mbar_arrive(&sh->unit_empty[slot]);
  }
  return u->f >= 0;
}

template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// The phase fraction of A keeps all its bits here (cis_q32).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
umma_contract_pairs(const FrameIO* __restrict__ frames, Consts k, Geo g, int out_dtype, unsigned* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* stages = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  PixStage* pix = (PixStage*)(stages + kStages * kStageBytes);
  Shared* sh = (Shared*)(pix + kPixStages);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t rank;  // in the pair; the CTA of rank 0 leads: its MMA thread drives both
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&sh->full[i], kAWarps + 1 + (rank == 0 ? 1 : 0));  // producer warps, B, the peer
      mbar_init(&sh->empty[i], 1);
    }
    for (int i = 0; i < kPixStages; ++i) {
      mbar_init(&sh->pix_full[i], 1);
      mbar_init(&sh->pix_empty[i], kAWarps);
    }
    for (int i = 0; i < kUnitSlots; ++i) {
      mbar_init(&sh->unit_full[i], 1);
      mbar_init(&sh->unit_empty[i], kAWarps + kSumWarps + 2);  // + the MMA (or relay) thread, the B loader
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->acc_full[i], 1);
      mbar_init(&sh->acc_empty[i], 2 * kSumWarps);
    }
    mbar_init(&sh->fin, 1);
    sh->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (g.NH != g.NT) {
    // the images end at row NT of a half: zeros in the 8 rows that the MMA reads beyond it
    for (int i = threadIdx.x; i < kStages * 2 * 64; i += kThreads)
      *reinterpret_cast<uint4*>(stages + (i >> 7) * kStageBytes + (2 + ((i >> 6) & 1)) * kPartBytes + g.NT * 128 +
                                (i & 63) * 16) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  cluster_sync();  // the peer's barriers exist
  fence_after();
  wait_prior_grid();  // the operand builder's writes are visible
  const uint32_t tmem = sh->tmem_base;
  const int64_t rows_total = (int64_t)k.V * k.Ns;

  if (warp < kAWarps) {
    // ------- A producers: thread = accumulator row, kAPx pixels of every stage -------
    // A entries of padded pixels and of rows past the cube need no masking: the B image
    // rows of padded pixels are zero, and rows past the cube are never written out.
    regs_dec<kRegsA>();
    const int quarter = warp & 3, part = warp >> 2;
    const int r = quarter * 32 + lane;
    const int j0 = part * kAPx;
    // this thread's A row; its 16-byte units sit at (unit ^ (row & 7)), the 128-byte swizzle
    unsigned char* arow = stages + r * 128;
    uint32_t st = 0, ph = 0, ps = 0, pph = 0, ui = 0;
    Unit x;
    bool alive = true;
    while (alive && next_unit(sh, ui++, status, &x, true)) {
      const int64_t gr = (int64_t)x.mt * 128 + r;
      const bool row_ok = gr < rows_total;
      const int v = row_ok ? (int)(gr / k.Ns) : x.v_first;
      const uint32_t n = row_ok ? (uint32_t)(gr % k.Ns) : 0u;
      // the row's phases: in the ring (the tile's channels, kPixChunks chunks a slot), or in
      // global memory when the tile spans more channels than the ring holds
      const bool staged = x.span <= kMaxCh;
      const uint32_t vl = row_ok ? v - x.v_first : 0;
      const FrameIO& fr = frames[x.f];
      const int64_t row_at = (int64_t)(row_ok ? v : 0) * fr.Pcap + (int64_t)x.c0 * kChunkPx + j0;
      const uint32_t chunks = x.c1 - x.c0;
      uint32_t cyc[kAPx];
      auto fetch = [&](uint32_t i) -> bool {  // the phases of the unit's stage i
        const uint32_t sub = i % kPixChunks;
        if (sub == 0 && !warp_wait(&sh->pix_full[ps], pph, sh, status)) return false;
        const uint32_t* pa = staged ? &pix[ps].a[vl][sub * kChunkPx + j0] : fr.phA + row_at + i * kChunkPx;
        const uint32_t* pc = staged ? &pix[ps].c[vl][sub * kChunkPx + j0] : fr.phC + row_at + i * kChunkPx;
#pragma unroll
        for (int j4 = 0; j4 < kAPx; j4 += 4) {
          const uint4 a4 = *reinterpret_cast<const uint4*>(pa + j4);
          const uint4 c4 = *reinterpret_cast<const uint4*>(pc + j4);
          cyc[j4] = a4.x * n + c4.x;
          cyc[j4 + 1] = a4.y * n + c4.y;
          cyc[j4 + 2] = a4.z * n + c4.z;
          cyc[j4 + 3] = a4.w * n + c4.w;
        }
        if (sub == kPixChunks - 1 || i == chunks - 1) {
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->pix_empty[ps]);
          if (++ps == kPixStages) ps = 0, pph ^= 1u;
        }
        return true;
      };
      if (chunks > 0) alive = fetch(0);
      bool free_now = false;  // the next stage's slot was seen free
      for (uint32_t i = 0; alive && i < chunks; ++i) {
        if (!__all_sync(0xffffffffu, free_now) && !warp_wait(&sh->empty[st], ph ^ 1u, sh, status)) {
          alive = false;
          break;
        }
        unsigned char* at = arow + st * kStageBytes;
#pragma unroll
        for (int j4 = 0; j4 < kAPx; j4 += 4) {
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const float2 f = cis_q32(cyc[j4 + t]);
            split2<0>(f.x, f.y, hi[t], lo[t]);
          }
          unsigned char* unit = at + (((part * 4 + j4 / 4) ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(unit) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(unit + kPartBytes) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        // the next stage's barrier is probed and its phases loaded while the stores land
        const uint32_t sn = st + 1 == kStages ? 0 : st + 1, pn = sn ? ph : ph ^ 1u;
        free_now = mbar_test(&sh->empty[sn], pn ^ 1u);
        if (i + 1 < chunks) alive = fetch(i + 1);
        // the MMAs read shared memory through the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->full[st]);
        st = sn, ph = pn;
      }
    }
  } else if (warp < kMmaWarp) {
    // ------- running sums: thread = accumulator row, every other 8 values of l -------
    // A finished group is added into registers (64 complex sums a thread at NT = 128) while
    // the MMAs fill the other accumulator; the sums leave for memory once per unit.
    regs_inc<kRegsSum>();
    const int quarter = warp & 3, half = (warp - kAWarps) >> 2;
    const int r = quarter * 32 + lane;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const uint64_t pol_p = policy_evict_last();
    uint32_t gi = 0;
    bool alive = true;
    for (uint32_t ui = 0; alive; ++ui) {
      // the unit's slot is given back after the write: read again there, not held in registers
      const uint32_t slot = ui % kUnitSlots;
      if (!warp_wait(&sh->unit_full[slot], (ui / kUnitSlots) & 1u, sh, status)) break;
      volatile Unit* xs = &sh->unit[slot];
      if (xs->f < 0) break;
      const uint32_t chunks = xs->c1 - xs->c0;
      const uint32_t ngr = unit_groups(chunks, xs->group);
      constexpr int kBlocks = kAccCols / 2 / 16;  // blocks of 8 values of l a warp may own
      float sre[kBlocks][8], sim[kBlocks][8];
#pragma unroll
      for (int b = 0; b < kBlocks; ++b)
#pragma unroll
        for (int i = 0; i < 8; ++i) sre[b][i] = sim[b][i] = 0.f;
      for (uint32_t gk = 0; gk < ngr; ++gk, ++gi) {
        if (!warp_wait(&sh->acc_full[gi & 1u], (gi >> 1) & 1u, sh, status)) {
          alive = false;
          break;
        }
        fence_after();
        if (chunks > 0) {
          const uint32_t acc = tmem + lane_base + (gi & 1u) * kAccCols;
#pragma unroll
          for (int b = 0; b < kBlocks; ++b) {
            const int jb = half * 8 + b * 16;
            if (jb < g.NT) {
              uint32_t re[8], im[8];
              tmem_ld8(acc + jb, re);
              tmem_ld8(acc + g.NH + jb, im);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                sre[b][i] += __uint_as_float(re[i]);
                sim[b][i] += __uint_as_float(im[i]);
              }
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_at(&sh->acc_empty[gi & 1u], 0);
      }
      if (!alive) break;
      // (a group of one at the end of a unit of two-chunk groups: at most 2e-8 of its sums)
      const float lost = xs->group > 1 ? kShort2 : kShort1;
      auto whole = [lost](float x) { return fmaf(x, lost, x); };
      const int mt = xs->mt, nt = xs->nt;
      const FrameIO& fr = frames[xs->f];
      const int64_t gr = (int64_t)mt * 128 + r;
      if (gr >= rows_total) {
        // a row past the cube: nothing to write
      } else if (g.direct) {
        const float2 oscale = sigma_unscale(fr, sigma_scaling(kTierFp32Tensor));
#pragma unroll
        for (int b = 0; b < kBlocks; ++b) {
          const int jb = half * 8 + b * 16;
          if (jb >= g.NT) continue;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int l = nt * g.NT + jb + i;
            if (l < k.L) {
              const int64_t o = gr * k.L + l;
              const float re = whole(sre[b][i]) * oscale.x * oscale.y, im = whole(sim[b][i]) * oscale.x * oscale.y;
              if (out_dtype == RSIM_C128)
                reinterpret_cast<double2*>(fr.cube)[o] = make_double2((double)re, (double)im);
              else
                reinterpret_cast<float2*>(fr.cube)[o] = make_float2(re, im);
            }
          }
        }
      } else {
        // tiled partial sums: column pair p of accumulator row r is float4 p * 128 + r of
        // the tile, so the warp's 32 rows write 512 contiguous bytes.  Columns past L
        // (last column tile) land in the tile's padding and are never read.
        float4* t4 = reinterpret_cast<float4*>(fr.partial + (int64_t)xs->s * g.sstride +
                                               ((int64_t)mt * g.ntiles + nt) * (128 * g.NT)) + r;
#pragma unroll
        for (int b = 0; b < kBlocks; ++b) {
          const int jb = half * 8 + b * 16;
          if (jb >= g.NT) continue;
#pragma unroll
          for (int i = 0; i < 8; i += 2)
            st_hint_v4(t4 + ((jb + i) >> 1) * 128,
                       make_float4(whole(sre[b][i]), whole(sim[b][i]), whole(sre[b][i + 1]), whole(sim[b][i + 1])),
                       pol_p);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->unit_empty[slot]);
    }
  } else {
    regs_dec<kRegsRest>();
    if (warp == kMmaWarp) {
      if (lane == 0 && rank == 0) {
        // ------------- leader: MMA issuer (one thread) -------------
        uint32_t st = 0, ph = 0, gi = 0, ui = 0;
        Unit x;
        bool alive = true;
        const uint32_t idesc = idesc_f16(2 * g.NH);
        const uint64_t desc0 = sdesc_sw128(smem_u32(stages));  // hi A of stage 0
        while (alive && next_unit(sh, ui++, status, &x, false)) {
          const uint32_t chunks = x.c1 - x.c0;
          const uint32_t ngr = unit_groups(chunks, x.group);
          for (uint32_t gk = 0; gk < ngr; ++gk, ++gi) {
            const uint32_t n = group_chunks_of(chunks, ngr, gk);
            const uint32_t acc = tmem + (gi & 1u) * kAccCols;
            if (!mbar_wait(&sh->acc_empty[gi & 1u], ((gi >> 1) & 1u) ^ 1u, sh, status)) {
              alive = false;
              break;
            }
            fence_after();
            for (uint32_t c = 0; c < n; ++c) {
              if (!mbar_wait(&sh->full[st], ph, sh, status)) {
                alive = false;
                break;
              }
              fence_after();
              const uint64_t a = desc0 + (uint64_t)(st * (kStageBytes >> 4));
              mma_stage(acc, a, a + (uint64_t)(2 * (kPartBytes >> 4)), idesc, c);
              mma_commit(&sh->empty[st]);
              if (++st == kStages) st = 0, ph ^= 1u;
            }
            if (!alive) break;
            if (n > 0) {
              mma_commit(&sh->acc_full[gi & 1u]);
            } else {
              mbar_arrive(&sh->acc_full[gi & 1u]);
              mbar_arrive_at(&sh->acc_full[gi & 1u], 1);
            }
          }
        }
        // every issued MMA (and every earlier commit) completes before either CTA leaves
        mma_commit(&sh->fin);
        mbar_wait(&sh->fin, 0, sh, status);
      } else if (lane == 0) {
        // ------------- peer: passes on that its part of a stage is there -------------
        uint32_t st = 0, ph = 0, ui = 0;
        Unit x;
        bool alive = true;
        while (alive && next_unit(sh, ui++, status, &x, false)) {
          for (uint32_t c = x.c0; c < x.c1; ++c) {
            if (!mbar_wait(&sh->full[st], ph, sh, status)) {
              alive = false;
              break;
            }
            mbar_arrive_at(&sh->full[st], 0);
            if (++st == kStages) st = 0, ph ^= 1u;
          }
        }
        mbar_wait(&sh->fin, 0, sh, status);
      }
    } else if (warp == kMmaWarp + 1) {
      // ------------- pixel loader: work units + bulk copies of the tile's phases -------------
      if (lane == 0) {
        uint32_t ps = 0, pph = 0;
        int u = pair;
        for (uint32_t ui = 0;; ++ui, u += pairs) {
          Unit x;
          x.f = -1;
          if (u < g.total_units) x = decode(g, frames, k, u, (int)rank);
          const uint32_t slot = ui % kUnitSlots, uph = (ui / kUnitSlots) & 1u;
          if (!mbar_wait(&sh->unit_empty[slot], uph ^ 1u, sh, status)) break;
          sh->unit[slot] = x;
          mbar_arrive(&sh->unit_full[slot]);
          if (x.f < 0) break;
          const FrameIO& fr = frames[x.f];
          const bool staged = x.span > 0 && x.span <= kMaxCh;
          bool alive = true;
          for (uint32_t c = x.c0; c < x.c1; c += kPixChunks) {
            if (!mbar_wait(&sh->pix_empty[ps], pph ^ 1u, sh, status)) {
              alive = false;
              break;
            }
            if (staged) {
              const uint32_t bytes = 4u * kChunkPx * (x.c1 - c < kPixChunks ? x.c1 - c : kPixChunks);
              mbar_expect_tx(&sh->pix_full[ps], 2u * bytes * x.span);
              for (int i = 0; i < x.span; ++i) {
                const int64_t ro = (int64_t)(x.v_first + i) * fr.Pcap + (int64_t)c * kChunkPx;
                bulk_g2s(pix[ps].a[i], fr.phA + ro, bytes, &sh->pix_full[ps]);
                bulk_g2s(pix[ps].c[i], fr.phC + ro, bytes, &sh->pix_full[ps]);
              }
            } else {
              mbar_arrive(&sh->pix_full[ps]);
            }
            if (++ps == kPixStages) ps = 0, pph ^= 1u;
          }
          if (!alive) break;
        }
      }
    } else if (warp == kMmaWarp + 2) {
      // ------------- B loader: bulk copies of this CTA's half of a chunk's B images -------------
      // rank 0: the re-rows (the accumulator's first NH columns), rank 1: the im-rows
      if (lane == 0) {
        const uint64_t pol_b = policy_evict_first();
        const uint32_t half = (uint32_t)g.NT * 128u;
        uint32_t st = 0, ph = 0, ui = 0;
        Unit x;
        bool alive = true;
        while (alive && next_unit(sh, ui++, status, &x, false)) {
          const FrameIO& fr = frames[x.f];
          for (uint32_t c = x.c0; c < x.c1; ++c) {
            if (!mbar_wait(&sh->empty[st], ph ^ 1u, sh, status)) {
              alive = false;
              break;
            }
            const unsigned char* src = fr.bimg + ((int64_t)x.nt * fr.bimg_nch + c) * 4 * half + rank * half;
            unsigned char* dst = stages + st * kStageBytes + 2 * kPartBytes;
            uint64_t* bar = &sh->full[st];
            mbar_expect_tx(bar, 2 * half);
            bulk_g2s_hint(dst, src, half, bar, pol_b);
            bulk_g2s_hint(dst + kPartBytes, src + 2 * half, half, bar, pol_b);
            if (++st == kStages) st = 0, ph ^= 1u;
          }
        }
      }
    }
  }

  __syncwarp();
  if (threadIdx.x == 0 && *(volatile int*)&sh->abort) {
    // a wait ran out: give the bulk copies in flight a millisecond to land
    const uint64_t t0 = globaltimer();
    while (globaltimer() - t0 < 1000000ull) {
    }
  }
  fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other may still signal it
  if (warp == kMmaWarp) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

}  // namespace

cudaError_t launch_umma_pairs(const Consts& k, const FrameIO* frames, int F, int splits, int nt, bool use_partial,
                              int grid, int num_sms, int64_t nch_max, int out_dtype, const int32_t* order,
                              unsigned* status, cudaStream_t st) {
  const int64_t rows = (int64_t)k.V * k.Ns;
  Geo g;
  g.NT = nt;
  g.NH = (nt + 15) / 16 * 16;  // N = 2 NH is a multiple of 32
  g.ntiles = (k.L + nt - 1) / nt;
  g.mpairs = (int)((rows + 255) / 256);
  g.splits = splits;
  g.direct = use_partial ? 0 : 1;
  g.F = F;
  g.sstride = tensor_split_stride(k.V, k.Ns, k.L, nt);
  g.order = order;
  const int64_t upf = (int64_t)g.mpairs * g.ntiles * splits;
  if (upf * F > 0x7FFFFFFF - num_sms) return cudaErrorInvalidValue;  // unit numbers are ints
  g.upf = (int)upf;
  g.total_units = g.upf * F;
  // persistent pairs, one CTA per SM (shared memory and tensor memory allow no more), that
  // take every (number of pairs)-th unit
  int pairs = std::max((grid > 0 ? std::min(grid, num_sms) : num_sms) / 2, 1);
  // A call of more than about 2 ms (0.85 us a chunk) does not hold the SMs to its end: its
  // pairs take about 0.25 ms of units each and leave, so that the blocks of a short request
  // on a stream of higher priority get in between (a pair's start costs a few us).
  const double unit_us = 0.85 * (double)nch_max / splits;
  if (grid == 0 && unit_us * g.total_units > 2000.0 * pairs) {
    const int per = (int)std::max(1.0, 250.0 / std::max(unit_us, 1.0));
    pairs = std::max(pairs, (g.total_units + per - 1) / per);
  }
  pairs = std::min(pairs, g.total_units);
  const int smem = kStages * kStageBytes + kPixStages * (int)sizeof(PixStage) + (int)sizeof(Shared) + 1024;
  const cudaError_t e =
      cudaFuncSetAttribute(umma_contract_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(umma_contract_pairs, dim3(2 * pairs), dim3(kThreads), (size_t)smem, st, frames, k, g,
                          out_dtype, status);
}

}  // namespace rsim
