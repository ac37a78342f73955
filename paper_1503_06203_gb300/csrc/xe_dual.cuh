// The correlator kernel of product path 1 at its default share: the tensor
// pipe and the dp4a pipe of every SM sub-partition driven by warps of their own.
//
// Both pipes multiply int8 at about the same rate on this GPU (64 products a
// cycle and sub-partition) and run side by side, so each takes about half of
// every 128-sample chunk of a 64 x 64 tile. What bounds a kernel that uses
// both is neither pipe but what feeds them:
// - Operand loads. One warp running both pipes on a 16 x 16 piece
//   (chunk_hybrid in xe_corr.cuh: 96 registers, 24 of them sums) loads 6 words
//   per 8 dp4a and keeps the shared-memory data path 77% busy; here a dp4a
//   thread owns an 8 x 8 micro-tile of one product (16 words per 64 dp4a) and
//   an MMA warp a 32 x 16 piece (55% busy), which is what the register split
//   below is for.
// - Instruction fetch. Straight dp4a code runs at full rate from loops of up to
//   32 KB (the SM's instruction cache, all roles together) and 1.6x slower
//   beyond; the first form of this kernel, unrolled to 137 KB, was slower than
//   the kernel it replaces. So the loops below stay rolled.
// - Issue slots: an int8 MMA takes 5 and a chunk's unpack about 500 a warp.
//
// Measured against the kernel that ran both pipes in every product warp, whole
// passes: N=256, F=256, T=16384 5019 -> 4220 us (220 -> 262 effective TOPS);
// N=8192, F=4, T=2048 9440 -> 7964 us; N=1024, F=64, T=4096 4733 -> 3977 us
// (schedules the same). Now: tensor pipe 79%, dp4a's pipe 63%, issue 62%.
//
// Roles (512 threads, one CTA per SM, launched with 128 registers a thread,
// then re-split by setmaxnreg: 2 x 104 + 216 + 88 = 512 a lane):
//   warps 0-7   tensor cores: the first 64 or 96 samples of each chunk, P1, P2
//               and Q of a 32 x 16 piece each (48 sums), two warps per
//               sub-partition (one cannot hide its own fragment loads: 80
//               against 68 cycles an MMA);
//   warps 8-11  dp4a: the chunk's other samples. Warp w = 2 q + h takes columns
//               8 m + 4 h + (0..3) of all 64 rows: P1 (q = 0) or P2 (q = 1)
//               over its samples, and Q over half of them, so the four warps
//               carry equal work with two 8 x 8 micro-tiles of sums each (128
//               registers), operands double-buffered 8 samples ahead;
//   warps 12-15 TMA issue and unpack. ldmatrix transposes the bytes (sm_103a's
//               16 x 16 byte form), so a 16-byte vector of samples of an
//               element takes half a load instruction and no byte permutes:
//               about 180 instructions a warp and box, where loading row words
//               and permuting took 230. Every one of them delays the dp4a warp
//               that shares its issue port: N=8192 (F=1, T=2048) 2009 -> 1939
//               us, N=256 (F=152, T=4096) 654 -> 638 us with the shares below
//               re-tuned.
// At the end of an item the dp4a warps fold their sums into (Re, Im) parts and
// add them into a tile in shared memory; the tensor warps add theirs and write
// the packed triangle from it, in whole 128-byte runs of a row.
#pragma once
#include "xe_corr.cuh"

namespace xe {

constexpr int kDualStages = 3;
constexpr int kDualBufs = 3;
constexpr int kDualMmaWarps = 8;
constexpr int kDualDpWarps = 4;
constexpr int kDualUnpackWarp = kDualMmaWarps + kDualDpWarps;
constexpr int kDualThreads = (kDualUnpackWarp + 4) * 32;
// Of every 8 chunks, those whose first 96 samples run on the tensor cores and
// the last 32 on dp4a (the others: 64 and 64), off and on the diagonal.
// Measured at 1, 2, 3 and 4 off it: N=8192 2001, 1939, 1977 and 2046 us (F=1,
// T=2048). On it (where dp4a skips more of the tile than the MMA's granularity
// lets the tensor cores skip) at 0, 1 and 2: N=64 213, 206 and 211 us (F=152,
// T=16384), N=256 646, 638 and 638 us (F=152, T=4096).
constexpr uint32_t kThreeOff = 2, kThreeDiag = 1;
constexpr int kRegsLaunch = 128, kRegsMma = 104, kRegsDp = 216, kRegsUnpack = 88;
static_assert(2 * kRegsMma + kRegsDp + kRegsUnpack <= 4 * kRegsLaunch, "setmaxnreg draws on the launch's registers");

// What the roles need to know of a chunk: written by the TMA issuer beside the
// box, passed on by the unpack warps beside the planes. The first 16 bytes are
// read with one load, the rest only for masked chunks and at an item's end.
struct __align__(16) DualMeta {
  int32_t flags;  // kMetaValid | kMetaEnd | kMetaMasked | write mode << 4 | tensor-core k-steps << 8
  int32_t bij;    // bi | bj << 16
  int32_t rows;   // samples past this one count as zero
  int32_t f;      // band
  int32_t lo, hi; // masked chunks: valid samples [lo, hi)
  int64_t B;
  int32_t* vis;
  int32_t N;
};
enum : int { kMetaMasked = 8 };

// (1024: the boxes' TMA swizzle follows the address)
constexpr uint32_t kDualAlign = 1024;

struct __align__(128) DualSmem {
  uint8_t box[kDualStages][2][kBoxBytes];          // TMA ring: [stage][A|B][time][element], 64-byte swizzle
  uint8_t plane[kDualBufs][2][3][kPlaneBytes];     // [buffer][A|B][slot][element][time]
  int32_t part[2][kTile * kTile];                  // Re and Im of the item under way, swizzled (part_at)
  DualMeta meta[kDualStages], pmeta[kDualBufs];    // (from part to here: zero at first, clear_smem)
  uint64_t full[kDualStages], bempty[kDualStages]; // box landed / read by the 4 unpack warps
  uint64_t pfull[kDualBufs], pempty[kDualBufs];    // planes written / read by the 12 product warps
  uint64_t mfull, mempty;                          // dp4a parts added; item written and `part` zero again
};

// Thread k of n's share of the zeroes a CTA starts with: no sums, and no chunk
// in any buffer. The dp4a warps read a buffer's meta, and load operands at the
// offset it names, also when the wait for it ran out, so it must never be what
// shared memory happened to hold. (Not reading it then took 0.5% of every
// frame, thread 0 clearing it 1%: the loops' code changes with either.)
__host__ __device__ __forceinline__ void clear_smem(DualSmem& sm, int k, int n) {
  constexpr int kWords = (sizeof(sm.part) + sizeof(sm.meta) + sizeof(sm.pmeta)) / 4;
  int32_t* const p = sm.part[0];
  for (; k < kWords; k += n) p[k] = 0;
}

// Hides a value's origin from the compiler, which would otherwise split the
// first or last iteration off the loops below and double their code.
__device__ __forceinline__ void opaque(uint32_t& v) { asm volatile("" : "+r"(v)); }

template <int n>
__device__ __forceinline__ void regs_up() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(n));
}
template <int n>
__device__ __forceinline__ void regs_down() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(n));
}

// Index of entry (row, col) in DualSmem::part[0 or 1]. The rows of a warp's
// 8 x 4 lane block (dp4a) fall on different 16-byte groups, so its adds are
// free of bank conflicts.
__device__ __forceinline__ int part_at(int row, int col) { return row * kTile + (col ^ ((row & 7) << 2)); }

// ---- tensor-core side -----------------------------------------------------------
struct MmaFrag {
  uint32_t a[2][4], b0[4], b1[2];
};

// Shared-memory offsets of a warp's fragments within a plane (k-step 0); the
// two slots are the piece's row halves on a full tile, and a 16 x 16 piece
// plus (warps 0-3) a single 16 x 8 sub-tile on a diagonal one.
struct MmaPiece {
  uint32_t a[2], b0, b1;
};

template <bool kDiag>
__device__ __forceinline__ void mma_load(uint32_t pa, uint32_t pb, const MmaPiece& p, uint32_t kx, bool single,
                                         MmaFrag& f) {
  ldsm_x4(pa + (p.a[0] ^ kx), f.a[0][0], f.a[0][1], f.a[0][2], f.a[0][3]);
  if (!kDiag || single) ldsm_x4(pa + (p.a[1] ^ kx), f.a[1][0], f.a[1][1], f.a[1][2], f.a[1][3]);
  ldsm_x4(pb + (p.b0 ^ kx), f.b0[0], f.b0[1], f.b0[2], f.b0[3]);
  if (kDiag && single) ldsm_x2(pb + (p.b1 ^ kx), f.b1[0], f.b1[1]);
}

// k-steps [0, ks) of the chunk. The other warp of the sub-partition covers the
// fragment loads' latency.
template <bool kDiag>
__device__ __forceinline__ void mma_chunk(uint32_t a_base, uint32_t b01, uint32_t b2, const MmaPiece& p, int ks,
                                          bool single, int32_t (&acc)[3][2][2][4]) {
  uint32_t kx = 0;
#pragma unroll 1
  for (int k = 0; k < ks; ++k, kx += 32) {
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) {
      MmaFrag c;
      mma_load<kDiag>(a_base + pl * kPlaneBytes, pl < 2 ? b01 + pl * kPlaneBytes : b2, p, kx, single, c);
      int32_t(&s)[2][2][4] = acc[pl];
      mma_s8_16832(s[0][0], c.a[0][0], c.a[0][1], c.a[0][2], c.a[0][3], c.b0[0], c.b0[1]);
      mma_s8_16832(s[0][1], c.a[0][0], c.a[0][1], c.a[0][2], c.a[0][3], c.b0[2], c.b0[3]);
      if (!kDiag) {
        mma_s8_16832(s[1][0], c.a[1][0], c.a[1][1], c.a[1][2], c.a[1][3], c.b0[0], c.b0[1]);
        mma_s8_16832(s[1][1], c.a[1][0], c.a[1][1], c.a[1][2], c.a[1][3], c.b0[2], c.b0[3]);
      } else if (single) {
        mma_s8_16832(s[1][0], c.a[1][0], c.a[1][1], c.a[1][2], c.a[1][3], c.b1[0], c.b1[1]);
      }
    }
  }
}

// Diagonal tile: the 20 sub-tiles of 16 x 8 that hold entries with i <= j are
// eight 16 x 16 pieces for warps 0-7 and the four sub-tiles of pieces (2, 2)
// and (3, 3) for warps 0-3: 5 sub-tiles per sub-partition (warps w, w + 4).
__device__ __forceinline__ void diag_piece(int w, int& pr, int& pc) {
  pr = (0x9500 >> (2 * w)) & 3;   // 0 0 0 0 1 1 1 2
  pc = (0xF9E4 >> (2 * w)) & 3;   // 0 1 2 3 1 2 3 3
}

// Adds a 16 x 8 sub-tile of the tensor-core sums, folded to (Re, Im), to the dp4a parts.
__device__ __forceinline__ void add_subtile(int32_t* part, int row0, int col0, int lane, const int32_t* p1,
                                            const int32_t* p2, const int32_t* qq) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int at = part_at(row0 + (lane >> 2) + 8 * h, col0 + 2 * (lane & 3));
    int2* re = reinterpret_cast<int2*>(part + at);
    int2* im = reinterpret_cast<int2*>(part + kTile * kTile + at);
    uint2 vr = *reinterpret_cast<uint2*>(re), vi = *reinterpret_cast<uint2*>(im);
    const uint32_t a0 = p1[2 * h], a1 = p1[2 * h + 1], b0 = p2[2 * h], b1 = p2[2 * h + 1];
    vr.x += a0 + b0;
    vr.y += a1 + b1;
    vi.x += static_cast<uint32_t>(qq[2 * h]) - a0 + b0;
    vi.y += static_cast<uint32_t>(qq[2 * h + 1]) - a1 + b1;
    *reinterpret_cast<uint2*>(re) = vr;
    *reinterpret_cast<uint2*>(im) = vi;
  }
}

// Writes rows row0 .. row0 + 15, columns col0 .. col0 + ncol - 1 (ncol <= 16)
// of the item from `part` to the packed triangle and zeroes them there. A warp
// writes whole 128-byte runs of a row: lane = (column, Re or Im). fresh: store,
// else add (red: the same result, and nothing to wait for, whether or not
// other CTAs add to the tile). Entries with i > j or outside the N x N matrix
// are dropped; entry (i, j) lives at (p(i, j)) * 2, p(i, j) = i N - i(i-1)/2 + j - i.
// Lanes past ncol (a diagonal tile's 16 x 8 piece) touch nothing: their columns
// are another warp's or past `part`. One branch for the read and the zeroing;
// clamping the column instead took 1944 against 1934 us (N=8192, F=1, T=2048).
__device__ __forceinline__ void write_rows(int32_t* part, int N, int32_t* band, int i0, int j0, int row0, int col0,
                                           int ncol, int lane, bool store) {
  const int col = col0 + (lane >> 1), j = j0 + col;
  int32_t* src = part + (lane & 1) * (kTile * kTile);
  const int64_t i1 = i0 + row0;
  int32_t* dst = band + (i1 * N - i1 * (i1 - 1) / 2 - i1 + j) * 2 + (lane & 1);
  const bool live = (lane >> 1) < ncol && j < N;
#pragma unroll 1
  for (int r0 = 0; r0 < 16; r0 += 8) {
    int32_t v[8] = {};
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      int32_t* s = src + part_at(row0 + r0 + r, col);
      if ((lane >> 1) < ncol) {
        v[r] = *s;
        *s = 0;
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int i = i0 + row0 + r0 + r;
      if (live && j >= i && i < N) {
        if (store)
          *dst = v[r];
        else
          atomicAdd(dst, v[r]);
      }
      dst += 2 * (N - 1 - i);
    }
  }
}

// ---- dp4a side ------------------------------------------------------------------
struct DpFrag {
  uint32_t a[8][2], b[8][2];  // 8 samples of rows lr + 8k and of columns 8m + 4h + lc
};

__device__ __forceinline__ void dp_load(uint32_t ra, uint32_t rb, DpFrag& n) {
#pragma unroll
  for (int k = 0; k < 8; ++k) lds64(ra + 1024 * k, n.a[k][0], n.a[k][1]);
#pragma unroll
  for (int k = 0; k < 8; ++k) lds64(rb + 1024 * k, n.b[k][0], n.b[k][1]);
}

// 8 samples: loads the next operands (ra, rb) among the products of the
// current ones. On a diagonal tile only the 36 of 64 row/column block pairs
// with entries i <= j are computed. Off the diagonal the column side's two
// words sit swapped (unpack), so that a dp4a's two operands come from
// different register banks (without it N=8192, F=1, T=2048 takes 2001 us
// instead of 1925, N=256, F=256, T=16384 4317 instead of 4203).
template <bool kDiag>
__device__ __forceinline__ void dp_step(uint32_t ra, uint32_t rb, DpFrag& n, const DpFrag& f, int32_t (&acc)[8][8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u == 0)
        lds64(ra + 1024 * k, n.a[k][0], n.a[k][1]);
      else
        lds64(rb + 1024 * k, n.b[k][0], n.b[k][1]);
#pragma unroll
      for (int m = 0; m < 8; ++m)
        if (!kDiag || k <= m) dp4a_acc(acc[k][m], f.a[k][u], f.b[m][kDiag ? u : u ^ 1]);
    }
}

// Samples [first, end) of the chunk's main product (planes ra, rb) into acc,
// and `half` of them (from sq) of Q (planes qa, qb) into acq; then the next
// chunk's first operands. Addresses carry the lane's row and swizzle; XOR with
// a sample offset selects the samples. Loops of two steps (4.6 KB of code
// each): the roles' loops together must stay within the SM's 32 KB
// instruction cache, beyond which straight dp4a code runs 1.6x slower.
template <bool kDiag, typename Wait, typename Addr>
__device__ __forceinline__ void dp_chunk(uint32_t ra, uint32_t rb, uint32_t qa, uint32_t qb, uint32_t first,
                                         uint32_t end, uint32_t sq, uint32_t half, Wait next_chunk, Addr next_addr,
                                         DpFrag (&f)[2], int32_t (&acc)[8][8], int32_t (&acq)[8][8]) {
#pragma unroll 1
  for (uint32_t o = first; o < end; o += 16) {
    opaque(o);
    dp_step<kDiag>(ra ^ (o + 8), rb ^ (o + 8), f[1], f[0], acc);
    const bool last = o + 16 == end;
    dp_step<kDiag>(last ? qa ^ sq : ra ^ (o + 16), last ? qb ^ sq : rb ^ (o + 16), f[0], f[1], acc);
  }
  next_chunk();
#pragma unroll 1
  for (uint32_t o = sq; o < sq + half; o += 16) {
    opaque(o);
    dp_step<kDiag>(qa ^ (o + 8), qb ^ (o + 8), f[1], f[0], acq);
    uint32_t na = qa ^ (o + 16), nb = qb ^ (o + 16);
    if (o + 16 == sq + half) next_addr(na, nb);
    dp_step<kDiag>(na, nb, f[0], f[1], acq);
  }
}

// Fold: acc = P1 (sign -1) or P2 (sign +1), acq = part of Q; Re += acc and
// Im += acq + sign * acc in `part`, by shared-memory adds (four warps' shares
// of the same entries, in any order). Modulo 2^32; exact for in-range results.
__device__ __forceinline__ void dp_merge(int32_t* part, int lane, int col0, int sign, int32_t (&acc)[8][8],
                                         int32_t (&acq)[8][8]) {
  const int lr = lane >> 2, lc = col0 + (lane & 3);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const uint32_t at = smem_u32(part + part_at(lr, lc + 8 * m));
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      red_shared(at + k * (8 * kTile * 4), acc[k][m]);
      red_shared(at + k * (8 * kTile * 4) + kTile * kTile * 4, acq[k][m] + sign * acc[k][m]);
    }
  }
}

// The first 16 bytes of a chunk's meta.
__device__ __forceinline__ int4 meta_head(const DualMeta& m) { return *reinterpret_cast<const int4*>(&m); }

// ---- the kernel -----------------------------------------------------------------
template <int kMode>
__global__ void __launch_bounds__(kDualThreads, 1) corr_dual_kernel(const __grid_constant__ CUtensorMap tmap,
                                                                    CorrArgs args) {
  constexpr bool kFrames = kMode != kSingle;
  constexpr bool kHold = kMode == kGated;
  constexpr bool kArith = kMode == kGateArith;
  extern __shared__ uint8_t smem_raw[];
  // (aligned by an offset from smem_raw, so that the compiler keeps shared-space accesses)
  DualSmem& sm =
      *reinterpret_cast<DualSmem*>(smem_raw + ((kDualAlign - smem_u32(smem_raw) % kDualAlign) % kDualAlign));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kDualStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.bempty[s], kUnpackThreads / 32);
    }
    for (int b = 0; b < kDualBufs; ++b) {
      mbar_init(&sm.pfull[b], kUnpackThreads / 32);
      mbar_init(&sm.pempty[b], kDualMmaWarps + kDualDpWarps);
    }
    mbar_init(&sm.mfull, kDualDpWarps);
    mbar_init(&sm.mempty, kDualMmaWarps);
    fence_barrier_init();
  }
  clear_smem(sm, threadIdx.x, kDualThreads);
  // The next launch may set its CTAs up as these leave their SMs; a launch that
  // was allowed to do so waits here for everything before it in its stream.
  launch_dependents();
  wait_prerequisites();
  __syncthreads();

  if (warp >= kDualUnpackWarp) {
    // ================= unpack warps (+ TMA issue) =================
    regs_down<kRegsUnpack>();
    const int uw = warp - kDualUnpackWarp;  // 0..3
    const bool producer = uw == 0 && lane == 0;
    // The transpose is ldmatrix's: warp uw takes elements 16 uw .. + 15 of a box, and lane 4 g + q, from
    // four matrices of 16 samples (quads 16 q + 4 b .. + 3 as rows 4 q .. 4 q + 3 of matrix b), the 16
    // samples 16 q .. + 15 of elements g and g + 8, for samples 0..63 and 64..127. A row address is a
    // lane's own, so a quad pair that the planes hold swapped is read swapped (row_off[1]).
    const int row = lane & 15, bl = lane >> 4, rq = row >> 2;
    uint32_t row_off[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int t = 16 * rq + 4 * (bl ^ x) + (row & 3);
      row_off[x] = static_cast<uint32_t>(t * kTile + ((uw ^ ((t >> 1) & 3)) << 4));
    }
    const uint32_t out = (16 * uw + (lane >> 2)) * kTC + (((lane & 3) ^ plane_swz(lane >> 2)) << 4);
    Walk<kFrames, kHold, kArith> ld;
    uint32_t issued = 0;
    const CUtensorMap* fenced = nullptr;
    bool ended = false;
    // Issue the walk's current unit (chunk of an item) into ring slot s, or end
    // the chunk stream with an entry without kMetaValid (no copy).
    auto issue = [&](int s) {
      DualMeta& m = sm.meta[s];
      ++issued;
      if (!ld.valid()) {
        m.flags = 0;
        mbar_arrive(&sm.full[s]);
        ended = true;
        return;
      }
      const bool diag = ld.bi == ld.bj;
      const CUtensorMap* map = ld.map(&tmap);
      if (kFrames && map != fenced) {  // a frame descriptor copied in before the launch
        tensormap_acquire(map);
        fenced = map;
      }
      const int lo = kArith ? 0 : ld.T0 - ld.c * kTC;
      const int rows = kArith ? ld.gate_rows() : ld.T - ld.c * kTC;
      // k-steps of 32 samples that hold any; a full chunk alternates 2 and 3 on the tensor cores, a shorter
      // one gives dp4a its last one if it has more than one
      const int ksteps = (min(rows, kTC) + 31) >> 5;
      const uint32_t three = diag ? kThreeDiag : kThreeOff;
      const int mk = ksteps == 4 ? 2 + ((issued * three >> 3) - ((issued - 1) * three >> 3)) : max(1, ksteps - 1);
      int flags = kMetaValid | (mk << 8);
      if (lo > 0 || rows < kTC) {
        flags |= kMetaMasked;
        m.lo = lo;
        m.hi = rows;
      }
      if (ld.last() && !(kHold && ld.hold)) {  // the item is written after this chunk
        if constexpr (kFrames) {
          flags |= kMetaEnd | (ld.mode << 4);
          m.N = ld.fN;
          m.B = ld.fB;
          m.vis = ld.fvis;
        } else {
          flags |= kMetaEnd | ((ld.c0 == 0 && ld.c1 == ld.nch ? (args.fresh ? 0 : 1) : 2) << 4);
          m.N = args.N;
          m.B = args.B;
          m.vis = args.vis;
        }
      }
      *reinterpret_cast<int4*>(&m) = make_int4(flags, ld.bi | (ld.bj << 16), rows, ld.f);
      // (the arrive releases the stores above to the slot's waiters)
      mbar_arrive_expect_tx(&sm.full[s], diag ? kBoxBytes : 2 * kBoxBytes);
      const int t = kArith ? ld.c : ld.c * kTC;
      tma_load_3d(sm.box[s][0], map, &sm.full[s], ld.bi * kTile, ld.f, t);
      if (!diag) tma_load_3d(sm.box[s][1], map, &sm.full[s], ld.bj * kTile, ld.f, t);
    };
    if (producer) {
      if (!kFrames) tma_prefetch_desc(&tmap);
      ld.before(args);
    }
    uint32_t want = kDualStages;       // chunks to have issued before the current one is unpacked
    int is = 0;                        // ring slot of the next chunk to issue, and the phase its slot must have passed
    uint32_t isphase = 1, started = 0; // (the first pass over the ring finds it free)
    int s = 0, buf = 0;
    uint32_t sphase = 0, bphase = 1;   // (and over the buffers)
    for (;; ++want) {
      if (producer) {  // refill the slot that every unpack warp is done with (all of them, at first)
        while (!ended && issued < want) {
          opaque(started);
          if (started) {
            if (!mbar_wait_bounded(&sm.bempty[is], isphase, kSpinLimit)) {
              atomicOr(args.err, kErrTimeoutEmpty);
              ended = true;
              break;
            }
            issue(is);
            if (++is == kDualStages) {
              is = 0;
              isphase ^= 1;
            }
          }
          started = 1;
          ld.next();  // (its loads are under way while the next chunk is unpacked)
        }
      }
      if (!mbar_wait_bounded(&sm.pempty[buf], bphase, kSpinLimit) ||
          !mbar_wait_bounded(&sm.full[s], sphase, kSpinLimit)) {
        if (lane == 0) atomicOr(args.err, kErrTimeoutFull);
        break;
      }
      const DualMeta& m = sm.meta[s];
      const int4 head = meta_head(m);
      const int flags = head.x, bij = head.y;
      if (uw == 0 && lane == 0) {  // passed on with the planes
        *reinterpret_cast<int4*>(&sm.pmeta[buf]) = head;
        if (flags & kMetaEnd) {
          sm.pmeta[buf].B = m.B;
          sm.pmeta[buf].vis = m.vis;
          sm.pmeta[buf].N = m.N;
        }
      }
      if (!(flags & kMetaValid)) {
        if (lane == 0) mbar_arrive(&sm.pfull[buf]);
        break;
      }
      const bool diag = (bij & 0xFFFF) == (bij >> 16);
      if (flags & kMetaMasked) {  // rows outside [lo, hi) count as zero: blank what this warp unpacks of them
        const int lo = m.lo, hi = m.hi;
#pragma unroll 1
        for (int t = lane; t < kTC; t += 32)
          if (t < lo || t >= hi)
            for (int j = 0; j < (diag ? 1 : 2); ++j)
              *reinterpret_cast<uint4*>(sm.box[s][j] + t * kTile + ((uw ^ ((t >> 1) & 3)) << 4)) =
                  make_uint4(0x88888888u, 0x88888888u, 0x88888888u, 0x88888888u);
        __syncwarp();
        fence_proxy_async();  // before the slot's next copy
      }
      // a diagonal tile's column side is its row side, so its xr - xi comes from the same pass
#pragma unroll 1
      for (int j = 0; j < (diag ? 1 : 2); ++j) {
        const uint32_t box = smem_u32(sm.box[s][j]), pl = smem_u32(sm.plane[buf][j][0]);
        const uint32_t pld = j || diag ? smem_u32(sm.plane[buf][1][kPsd]) : 0u, pls = j ? 0u : pl + kPsd * kPlaneBytes;
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // samples 64 h .. 64 h + 63
          // the dp4a samples of an off-diagonal tile's column side: the two words of every 8 samples swapped
          const uint32_t at = box + (j && 2 * h + (rq >> 1) >= (flags >> 8) ? row_off[1] : row_off[0]) + 4096 * h;
          uint32_t wd[2][4];
          ldsm_t8_x2(at, wd[0][0], wd[1][0], wd[0][1], wd[1][1]);
          ldsm_t8_x2(at + 512, wd[0][2], wd[1][2], wd[0][3], wd[1][3]);
#pragma unroll
          for (int e = 0; e < 2; ++e) unpack_vec<false>(wd[e], (out ^ (64 * h)) + 1024 * e, pl, pl + kPlaneBytes, pls, pld);
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm.pfull[buf]);
        mbar_arrive(&sm.bempty[s]);
      }
      if (++s == kDualStages) {
        s = 0;
        sphase ^= 1;
      }
      if (++buf == kDualBufs) {
        buf = 0;
        bphase ^= 1;
      }
    }
    if (producer) {
      // Never leave with copies in flight (see xe_corr.cuh); the wait is bounded all the same.
      const uint32_t first = issued > kDualStages ? issued - kDualStages : 0;
      for (uint32_t k = first; k < issued; ++k)
        mbar_wait_bounded(&sm.full[k % kDualStages], (k / kDualStages) & 1, kSpinLimit);
    }
    return;
  }

  int32_t* const part = sm.part[0];
  int buf = 0;
  uint32_t phase = 0, items = 0;  // plane-buffer phase; items written so far

  if (warp < kDualMmaWarps) {
    // ================= tensor-core warps (and the writer) =================
    regs_down<kRegsMma>();
    int32_t acc[3][2][2][4];
#pragma unroll
    for (int k = 0; k < 48; ++k) (&acc[0][0][0][0])[k] = 0;
    const int l7 = lane & 7;
    const uint32_t xa = static_cast<uint32_t>((lane >> 4) ^ plane_swz(l7)) << 4;        // A: k half = lane / 16
    const uint32_t xb = static_cast<uint32_t>(((lane >> 3) & 1) ^ plane_swz(l7)) << 4;  // B: k half = (lane / 8) & 1
    const uint32_t arow = (lane & 15) * kTC + xa, brow = (l7 + ((lane >> 4) << 3)) * kTC + xb;
    int dr, dc;
    diag_piece(warp, dr, dc);
    const int sr = 2 + (warp >> 1), sn = warp & 1;  // single sub-tile (warps 0-3): piece (sr, sr), half sn
    for (;;) {
      if (!mbar_wait_bounded(&sm.pfull[buf], phase, kSpinLimit)) {
        if (lane == 0) atomicOr(args.err, kErrTimeoutFull);
        return;
      }
      const DualMeta& m = sm.pmeta[buf];
      const int4 head = meta_head(m);
      const int flags = head.x;
      if (!(flags & kMetaValid)) return;  // end of this CTA's chunks
      const int bi = head.y & 0xFFFF, bj = head.y >> 16;
      const bool diag = bi == bj;
      const int ks = min(flags >> 8, (head.z + 31) >> 5);
      const uint32_t a_base = smem_u32(sm.plane[buf][0][0]), b_side = smem_u32(sm.plane[buf][1][0]);
      const uint32_t b2 = b_side + kPsd * kPlaneBytes;
      if (ks > 0) {
        MmaPiece p;
        if (!diag) {
          p.a[0] = arow + (32 * (warp >> 2)) * kTC;
          p.a[1] = p.a[0] + 16 * kTC;
          p.b0 = brow + 16 * (warp & 3) * kTC;
          p.b1 = 0;
          mma_chunk<false>(a_base, b_side, b2, p, ks, true, acc);
        } else {
          p.a[0] = arow + 16 * dr * kTC;
          p.a[1] = arow + 16 * sr * kTC;
          p.b0 = brow + 16 * dc * kTC;
          p.b1 = l7 * kTC + xb + (16 * sr + 8 * sn) * kTC;
          mma_chunk<true>(a_base, a_base, b2, p, ks, warp < 4, acc);
        }
      }
      int32_t* band = nullptr;
      int N = 0;
      if (flags & kMetaEnd) {
        band = m.vis + static_cast<int64_t>(head.w) * m.B * 2;
        N = m.N;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.pempty[buf]);
      if (flags & kMetaEnd) {  // end of the item: add the dp4a parts and write it
        if (!mbar_wait_bounded(&sm.mfull, items & 1, kSpinLimit)) {
          if (lane == 0) atomicOr(args.err, kErrTimeoutFull);
          return;
        }
        const int mode = (flags >> 4) & 3, i0 = bi * kTile, j0 = bj * kTile;
        // the two slots of the piece: 16 rows each (a diagonal tile's second one: 8 columns, warps 0-3)
        const int row[2] = {diag ? 16 * dr : 32 * (warp >> 2), diag ? 16 * sr : 32 * (warp >> 2) + 16};
        const int col[2] = {diag ? 16 * dc : 16 * (warp & 3), diag ? 16 * sr + 8 * sn : 16 * (warp & 3)};
        const int slots = diag && warp >= 4 ? 1 : 2;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (r == slots) break;
          add_subtile(part, row[r], col[r], lane, acc[0][r][0], acc[1][r][0], acc[2][r][0]);
          if (r == 0 || !diag) add_subtile(part, row[r], col[r] + 8, lane, acc[0][r][1], acc[1][r][1], acc[2][r][1]);
        }
        __syncwarp();
#pragma unroll 1
        for (int r = 0; r < slots; ++r)
          write_rows(part, N, band, i0, j0, r ? row[1] : row[0], r ? col[1] : col[0], r && diag ? 8 : 16, lane, mode == 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.mempty);
        ++items;
#pragma unroll
        for (int k = 0; k < 48; ++k) (&acc[0][0][0][0])[k] = 0;  // (here, so that the sums' registers are free while writing)
      }
      if (++buf == kDualBufs) {
        buf = 0;
        phase ^= 1;
      }
    }
  }

  // ================= dp4a warps =================
  regs_up<kRegsDp>();
  int32_t acc[8][8], acq[8][8];
  uint32_t clear = 1;  // the next chunk begins an item
  const int q = (warp >> 1) & 1, h = warp & 1;
  const int lr = lane >> 2, lc = 4 * h + (lane & 3);
  // offsets of the lane's first row and column within a buffer's planes: main product and Q
  constexpr uint32_t kSide = 3 * kPlaneBytes, kBuf = 2 * kSide;
  const uint32_t ca = lr * kTC + (plane_swz(lr) << 4) + q * kPlaneBytes, cb = lc * kTC + (plane_swz(lc) << 4) + q * kPlaneBytes;
  const uint32_t cq = (kPsd - q) * kPlaneBytes;
  const uint32_t plane0 = smem_u32(sm.plane[0][0][0]);
  uint32_t base = plane0;
  DpFrag fr[2];
  if (!mbar_wait_bounded(&sm.pfull[0], 0, kSpinLimit)) {
    if (lane == 0) atomicOr(args.err, kErrTimeoutFull);
    return;
  }
  uint32_t primed = 0;  // fr[0] holds the current chunk's first operands
  int4 head = meta_head(sm.pmeta[0]);
  while (head.x & kMetaValid) {
    const bool diag = (head.y & 0xFFFF) == (head.y >> 16);
    const int nbuf = buf + 1 == kDualBufs ? 0 : buf + 1;
    const uint32_t nphase = nbuf ? phase : phase ^ 1;
    const uint32_t nbase = nbuf ? base + kBuf : plane0;
    const uint32_t ra = base + ca, rb = base + cb + (diag ? 0u : kSide);
    const uint32_t qa = ra + cq, qb = base + cb + kSide + cq;
    bool ok = true;
    opaque(clear);
    opaque(primed);
    if (clear) {
#pragma unroll
      for (int k = 0; k < 64; ++k) (&acc[0][0])[k] = (&acq[0][0])[k] = 0;
      clear = 0;
    }
    int4 next_head = head;
    auto next_chunk = [&](void) {  // waits for the next chunk's planes; its meta
      ok = mbar_wait_bounded(&sm.pfull[nbuf], nphase, kSpinLimit);
      next_head = meta_head(sm.pmeta[nbuf]);
    };
    // samples [first, end), whole k-steps; Q's half of them
    const uint32_t first = 32 * (head.x >> 8), end = min(kTC, (head.z + 31) & ~31), half = (end - first) / 2;
    if (head.z > static_cast<int>(first)) {
      if (!primed) dp_load(ra ^ first, rb ^ first, fr[0]);
      auto next_addr = [&](uint32_t& na, uint32_t& nb) {  // (if there is no next chunk, this one's: loaded, not used)
        const bool valid = next_head.x & kMetaValid;
        const bool xdiag = valid && (next_head.y & 0xFFFF) == (next_head.y >> 16);
        const uint32_t at = valid ? nbase : base, o = 32 * (next_head.x >> 8);
        na = (at + ca) ^ o;
        nb = (at + cb + (xdiag ? 0u : kSide)) ^ o;
      };
      if (diag)
        dp_chunk<true>(ra, rb, qa, qb, first, end, first + half * q, half, next_chunk, next_addr, fr, acc, acq);
      else
        dp_chunk<false>(ra, rb, qa, qb, first, end, first + half * q, half, next_chunk, next_addr, fr, acc, acq);
      primed = 1;
    } else {
      next_chunk();
      primed = 0;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.pempty[buf]);
    if (head.x & kMetaEnd) {
      // the previous item's parts must have been read
      if (!mbar_wait_bounded(&sm.mempty, (items & 1) ^ 1, kSpinLimit)) ok = false;
      if (ok) {
        dp_merge(part, lane, 4 * h, q ? 1 : -1, acc, acq);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.mfull);
        ++items;
        clear = 1;
      }
    }
    if (!ok) {
      if (lane == 0) atomicOr(args.err, kErrTimeoutFull);
      return;
    }
    head = next_head;
    buf = nbuf;
    base = nbase;
    phase = nphase;
  }
}

}  // namespace xe
