// Ground states of many sequences against every conformation on the tensor cores.
//
// A contact joins an even residue i and an odd residue j, so the score of sequence h on
// conformation s is a contraction over the residue pairs that are in contact in some conformation:
//   x_s(h) = sum_(i,j) K_s(i,j) e(h_i, h_j),   e = 0, 10, 23 for no, one or two H  (Table 1 x 10)
// with K_s the 0/1 contact matrix.  Every conformation of a box has the same number C of contacts,
// so e may be shifted by a constant: e - 10 is -10, 0 or 13, which (unlike 23) 8-bit floats (e4m3)
// hold exactly, and x = 10 C + sum K (e - 10).  All products and sums are whole numbers below 2^13,
// so the fp32 accumulators are exact.  One column of the contraction is constant (-10 against 0 for
// a conformation, 448 for the rows that pad the last tile, which puts those far below any score).
//
// scan_tc_kernel: persistent CTAs, one per SM, each a contiguous run of (256-sequence block,
// 256-conformation tile) units.  The block's features (2 x 128 rows) are written to shared memory by
// the epilogue warps; the conformations stream through a ring of stages of 8 KB slabs (256
// conformations x 32 pairs, stored in the order the tensor core reads them; one cp.async.bulk a stage).
// Both halves of the block use a slab while it is resident, which halves the L2 traffic per multiplication to
// 32 B/clk/SM (one half alone would need 64, more than L2 delivers to all SMs at once); while the
// tensor core works on one half's accumulator (256 TMEM columns) the epilogue drains the other's.
// The epilogue keeps per sequence the best score, the second best over groups of 32
// conformations (counted with multiplicity) and the first group that reaches the best: 16
// three-input maxima and five more instructions per 32 scores.
// A unit takes 2 x 128 clk per 32 pairs at the tensor cores' rate; each half has one accumulator, so a
// half's drain and hand-over (about 400 clk) overlap only the other half's multiplications.
// Measured (call, ids in L2): 16,384 ids of 3x3x3 160 us, the warp scan 13,600 us; 65,536 ids of 6x6
// 648 us, the pruned warp scan 6,600 us; floors at 128 clk per 128 x 256 x 32: 110 and 480 us.
//
// scan_tc_resolve: one warp per sequence merges the runs' results and scores the one group of 32
// conformations exactly, which gives the lowest minimiser, the tie and the energy gap.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "hp_internal.h"

namespace {

constexpr int kRows = 128;                 // sequences per accumulator (tensor-memory lanes)
constexpr int kBlock = 2 * kRows;          // sequences per block
constexpr int kTile = 256;                 // conformations per tile
constexpr int kGroup = 32;                 // conformations per group of the running best
constexpr int kSlabA = kRows * 32;         // bytes of 128 rows x 32 pairs
constexpr int kSlabB = kTile * 32;         // bytes of 256 conformations x 32 pairs
constexpr int kMaxSlots = 8;               // stages of the ring (at most)
constexpr int kMaxStage = 5;               // slabs per stage (at most)
constexpr int kEpiWarps = 16;             // four per tensor-memory lane quarter
constexpr int kParts = kEpiWarps / 4;     // column slices of a tile, one per epilogue warp of a quarter
constexpr int kCols = kTile / kParts;
constexpr int kThreads = 128 + 32 * kEpiWarps;  // producer, two issuers, one idle warp, epilogue
constexpr int kSmemMax = 226 * 1024;
constexpr uint32_t kSpin = 1u << 24;       // polls of a wait before it gives up
constexpr long long kChunk = 1ll << 19;    // sequences per launch (bounds the scratch: 27 MB)
constexpr size_t kMaxTable = 1ull << 30;   // largest conformation table
constexpr unsigned long long kPoolKeep = 32ull << 20;  // scratch that a library keeps on a device between calls
// e4m3: 13, -10, 1, 448
constexpr uint32_t kF13 = 0x55, kFm10 = 0xD2, kF1 = 0x38, kF448 = 0x7E;

struct TcParams {
  const uint8_t* tab;              // ntiles x nk slabs of kSlabB bytes
  const uint16_t* pairs;           // 32 nk entries: even index | odd index << 8; 0x1F1F (bits that are always
                                   // clear) for the constant and the unused columns
  const unsigned long long* ids;   // n ids, or NULL: base + row
  unsigned long long base;
  long long n, units;
  int nk, ntiles, cs, nslots;      // slabs per tile, tiles, slabs per stage of the ring, stages
  float* part;                     // [ctas + blocks][kParts][best, second, group][kBlock]
  unsigned* status;                // per CTA: 1 where its waits all succeeded
  uint32_t spin;
};

struct ResolveParams {
  TcParams t;
  int ctas;
  const uint32_t* rec;
  const int32_t* conf_class;
  int rec_words, NE, C, S_dir, T, prune;
  int32_t *phen, *aux, *gap;
  unsigned long long* counters;
  unsigned* err;                   // or NULL
};

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool poll(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok)
               : "r"(bar), "r"(parity)
               : "memory");
  return ok != 0;
}

// Bounded wait for a barrier phase; one that gives up raises the CTA's abort flag, which ends the
// other roles' waits too.
__device__ __noinline__ bool wait_phase(uint64_t* bar, uint32_t parity, volatile int* abort_flag, uint32_t limit) {
  const uint32_t b = sa(bar);
  for (uint32_t i = 0;; i++) {
    if (i >= limit) {
      *abort_flag = 1;
      return false;
    }
    if (poll(b, parity)) return true;
    if ((i & 255) == 255 && *abort_flag) return false;
  }
}

// The same by a converged warp for a barrier that is usually complete: one poll, then the loop.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, uint32_t limit) {
  if (limit != 0 && __all_sync(0xFFFFFFFFu, poll(sa(bar), parity))) return true;
  return __all_sync(0xFFFFFFFFu, wait_phase(bar, parity, abort_flag, limit));
}

__device__ __forceinline__ void drain(uint64_t* bar, uint32_t parity) {
  const uint32_t b = sa(bar);
  for (uint32_t i = 0; i < kSpin; i++)
    if (poll(b, parity)) return;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sa(bar)), "r"(n));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sa(bar)) : "memory");
}
// K-major operands without swizzle: core matrices of 8 rows x 16 bytes, the two of a 32-byte slab
// row 128 bytes apart, groups of 8 rows 256 bytes apart.  Low word of a slab's descriptor; the high
// word is the same for all.
__device__ __forceinline__ uint32_t slab_lo(uint32_t addr) { return (addr >> 4) | ((128u >> 4) << 16); }
constexpr uint32_t kSlabHi = (256u >> 4) | (1u << 14);
// e4m3 x e4m3 -> f32, both K-major, M 128, N 256
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kTile >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);

// One MMA of a slab pair / a commit, by one elected lane of a converged warp (always the same lane).
__device__ __forceinline__ void mma(uint32_t acc, uint32_t a, uint32_t b, bool accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 da, db;\n elect.sync _|q, 0xffffffff;\n setp.ne.u32 p, %5, 0;\n"
      " mov.b64 da, {%1, %3};\n mov.b64 db, {%2, %3};\n"
      " @q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %4, p;\n}\n" ::"r"(acc),
      "r"(a), "r"(b), "r"(kSlabHi), "r"(kIdesc), "r"((uint32_t)accumulate));
}
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile(
      "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(sa(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%"
      "21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]),
        "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]),
        "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
      : "r"(taddr));
}
// wait for the issued loads; v is tied to the wait so that no use is scheduled before it
__device__ __forceinline__ void tmem_wait(float (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]),
                 "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]),
                 "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]),
                 "+f"(v[30]), "+f"(v[31])
               :
               : "memory");
}

// even / odd residues of a sequence id (bit k = residue 2k / 2k + 1)
__device__ __forceinline__ uint32_t compress(unsigned long long g) {
  uint32_t r = 0;
#pragma unroll
  for (int k = 0; k < hp::kMaxHalf; k++) r |= (uint32_t)((g >> (2 * k)) & 1ull) << k;
  return r;
}
__device__ __forceinline__ unsigned long long id_of(const TcParams& p, long long row) {
  return p.ids ? p.ids[row] : p.base + (unsigned long long)row;
}
// first unit of CTA c; the CTA that holds unit u
__host__ __device__ __forceinline__ long long unit_begin(long long c, long long units, long long ctas) { return c * units / ctas; }
__host__ __device__ __forceinline__ long long cta_of(long long u, long long units, long long ctas) {
  return ((u + 1) * ctas - 1) / units;
}

__global__ void __launch_bounds__(kThreads, 1) scan_tc_kernel(const TcParams p) {
  extern __shared__ uint8_t tc_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_raw) + 127) & ~(uintptr_t)127);
  uint8_t* bring = smem + 2 * p.nk * kSlabA;
  __shared__ __align__(8) uint64_t full[kMaxSlots], empty[kMaxSlots], tfull[2], tempty[2], afull, done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sa(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nslots; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 2);
    }
    for (int h = 0; h < 2; h++) {
      mbar_init(&tfull[h], 1);
      mbar_init(&tempty[h], kEpiWarps);
    }
    mbar_init(&afull, kEpiWarps);
    mbar_init(&done, 2);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const long long u0 = unit_begin(blockIdx.x, p.units, gridDim.x), u1 = unit_begin(blockIdx.x + 1, p.units, gridDim.x);
  const int nk = p.nk;

  if (warp == 0 && lane == 0) {
    // ---------------------------------------------------------------- producer: conformation slabs
    uint32_t used[kMaxSlots];  // copies issued per stage (local memory: read only on the way out)
    for (int s = 0; s < kMaxSlots; s++) used[s] = 0;
    int slot = 0;
    uint32_t round = 0;
    bool ok = true;
    int tile = (int)(u0 % p.ntiles);
    for (long long u = u0; u < u1 && ok; u++) {
      const uint8_t* src = p.tab + (size_t)tile * nk * kSlabB;
      for (int k = 0; k < nk; k += p.cs) {
        if (!wait_phase(&empty[slot], (round & 1) ^ 1, abort_flag, p.spin)) {
          ok = false;
          break;
        }
        const uint32_t fb = sa(&full[slot]), bytes = (uint32_t)min(p.cs, nk - k) * kSlabB;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         sa(bring + slot * p.cs * kSlabB)),
                     "l"(src + k * kSlabB), "r"(bytes), "r"(fb)
                     : "memory");
        used[slot] = round + 1;
        if (++slot == p.nslots) {
          slot = 0;
          round++;
        }
      }
      if (++tile == p.ntiles) tile = 0;
    }
    // every copy has landed before the CTA may exit
    for (int s = 0; s < p.nslots; s++)
      if (used[s]) drain(&full[s], (used[s] - 1) & 1);
  } else if (warp == 1 || warp == 2) {
    // ---------------------------------------------------------------- MMA issuers, one per half
    // A wait on a barrier that is already complete costs the issuing warp about 200 clk, more than the
    // tensor core has queued; with an issuer per half one half's MMAs run during the other's waits
    // (one issuer for both halves: 999 instead of 723 us per 65,536 ids of 3x3x3 with the waits and stages
    // as they then were; 573 now).  The whole warp walks the loop and one elected lane issues, so that
    // addresses and descriptors stay in uniform registers.
    const int h = warp - 1;
    int slot = 0;
    uint32_t round = 0, seg = 0, uses = 0;
    bool ok = true;
    long long u = u0;
    const uint32_t a0 = slab_lo(sa(smem + h * nk * kSlabA)), b0 = slab_lo(sa(bring)), bstage = (uint32_t)(p.cs * kSlabB) >> 4;
    const uint32_t acc = tmem + h * kTile;
    while (u < u1 && ok) {
      const long long blk = u / p.ntiles, uend = min(u1, (blk + 1) * p.ntiles);
      const bool mine = h == 0 || p.n - blk * kBlock > kRows;  // else: only hand the stages back
      ok = warp_wait(&afull, seg & 1, abort_flag, p.spin);
      seg++;
      for (int left = (int)(uend - u); left > 0 && ok; left--) {
        uint32_t ad = a0;
        for (int k = 0; k < nk && ok; k += p.cs) {
          ok = warp_wait(&full[slot], round & 1, abort_flag, p.spin);
          // (after the stage: that wait then overlaps the epilogue's drain of this accumulator)
          if (k == 0 && mine && ok) {
            ok = warp_wait(&tempty[h], (uses & 1) ^ 1, abort_flag, p.spin);
            uses++;
          }
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t bd = b0 + slot * bstage;
          const int ke = min(p.cs, nk - k), freed = slot;
          if (++slot == p.nslots) {
            slot = 0;
            round++;
          }
          if (mine) {
#pragma unroll
            for (int i = 0; i < kMaxStage; i++)
              if (i < ke) mma(acc, ad + i * (kSlabA >> 4), bd + i * (kSlabB >> 4), k + i > 0);
          }
          ad += ke * (kSlabA >> 4);
          commit(&empty[freed]);
        }
        if (ok && mine) commit(&tfull[h]);
      }
      u = uend;
    }
    commit(&done);  // every MMA issued has finished before the tensor memory is freed
    drain(&done, 0);
  } else if (warp >= 4) {
    // ---------------------------------------------------------------- features and epilogue
    const int q = warp & 3;            // tensor-memory lane quarter this warp may read
    const int ch = (warp - 4) >> 2;    // columns kCols ch .. of each tile
    // row of the block whose features this thread writes, and which half of them
    const int frow = 32 * ((warp - 4) & 7) + lane, fhalf = (warp - 4) >> 3;
    uint32_t uses[2] = {0, 0};
    bool ok = true;
    long long u = u0;
    while (u < u1 && ok) {
      const long long blk = u / p.ntiles, uend = min(u1, (blk + 1) * p.ntiles);
      const int halves = p.n - blk * kBlock > kRows ? 2 : 1;
      // features of this segment's block; every MMA on the previous block has finished (its last
      // accumulators were waited for below)
      if (blk * kBlock + frow < p.n) {
        const unsigned long long g = id_of(p, blk * kBlock + frow);
        const uint32_t e = compress(g), o = compress(g >> 1);
        const int h = frow / kRows, r = frow % kRows;
        uint8_t* dst = smem + h * nk * kSlabA + (r >> 3) * 256 + (r & 7) * 16;
        for (int c = fhalf * nk; c < (fhalf + 1) * nk; c++) {  // 16 pairs at a time
          const uint4* pr = reinterpret_cast<const uint4*>(p.pairs + 16 * c);
          const uint4 pa = __ldg(pr), pb = __ldg(pr + 1);
          const uint32_t pw[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; i++) {
            w[i] = 0;
#pragma unroll
            for (int b = 0; b < 4; b++) {
              const uint32_t pair = (pw[2 * i + (b >> 1)] >> (16 * (b & 1))) & 0xFFFFu;
              // bits above residue 19 of either half are clear: an index of 31 reads 0
              const uint32_t x = (e >> (pair & 31u)) & 1u, y = (o >> ((pair >> 8) & 31u)) & 1u;
              w[i] |= ((x & y) * kF13 | ((x | y) ^ 1u) * kFm10) << (8 * b);
            }
          }
          *reinterpret_cast<uint4*>(dst + (c >> 1) * kSlabA + (c & 1) * 128) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&afull);
      float best[2] = {-1e30f, -1e30f}, sec[2] = {-1e30f, -1e30f};
      int grp[2] = {0, 0};
      for (; u < uend && ok; u++) {
        const int g0 = (int)(u - blk * p.ntiles) * (kTile / kGroup) + ch * (kCols / kGroup);
#pragma unroll
        for (int h = 0; h < 2; h++) {
          if (h >= halves || !ok) continue;
          ok = warp_wait(&tfull[h], uses[h] & 1, abort_flag, p.spin);
          if (!ok) continue;
          uses[h]++;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + h * kTile + ch * kCols;
          float v[2][32];
          tmem_ld32(ta, v[0]);
#pragma unroll
          for (int c = 0; c < kCols / kGroup; c++) {
            tmem_wait(v[c & 1]);
            if (c + 1 < kCols / kGroup) {
              tmem_ld32(ta + (c + 1) * kGroup, v[(c + 1) & 1]);
            } else {  // the accumulator is read: hand it back before the last maxima
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(&tempty[h]);
            }
            float(&x)[32] = v[c & 1];
            float m0 = fmaxf(fmaxf(x[0], x[1]), x[2]), m1 = fmaxf(fmaxf(x[3], x[4]), x[5]);
#pragma unroll
            for (int j = 6; j < 30; j += 4) {
              m0 = fmaxf(fmaxf(m0, x[j]), x[j + 1]);
              m1 = fmaxf(fmaxf(m1, x[j + 2]), x[j + 3]);
            }
            m0 = fmaxf(fmaxf(m0, x[30]), x[31]);
            const float m = fmaxf(m0, m1);
            sec[h] = fmaxf(sec[h], fminf(best[h], m));
            if (m > best[h]) grp[h] = g0 + c;
            best[h] = fmaxf(best[h], m);
          }
        }
      }
      float* out = p.part + ((size_t)(blockIdx.x + blk) * kParts + ch) * 3 * kBlock + 32 * q + lane;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        if (h >= halves) continue;
        out[h * kRows] = best[h];
        out[kBlock + h * kRows] = sec[h];
        out[2 * kBlock + h * kRows] = __int_as_float(grp[h]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  if (threadIdx.x == 0) p.status[blockIdx.x] = abort_word ? 0u : 1u;
}

// exact score of (e, o) on a conformation record
__device__ __forceinline__ int exact_score(const uint32_t* r, int NE, uint32_t e, uint32_t o) {
  const uint32_t *wo = r + NE, *we = r + NE + 3;
  int x = 10 * ((__popc(e & __ldg(we)) + __popc(o & __ldg(wo))) + 2 * (__popc(e & __ldg(we + 1)) + __popc(o & __ldg(wo + 1))) +
                4 * (__popc(e & __ldg(we + 2)) + __popc(o & __ldg(wo + 2))));
  for (uint32_t m = e; m; m &= m - 1) x += 3 * __popc(o & __ldg(r + (__ffs(m) - 1)));
  return x;
}

__global__ void __launch_bounds__(256) scan_tc_resolve(const ResolveParams p) {
  const TcParams& t = p.t;
  const int lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0 && p.counters) atomicAdd(p.counters, (unsigned long long)t.n * p.S_dir);
  const long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= t.n) return;
  const unsigned long long g = id_of(t, row);
  const uint32_t emask = (1u << p.NE) - 1u;
  const uint32_t e = compress(g) & emask, o = compress(g >> 1);
  const long long blk = row / kBlock;
  const int r = (int)(row % kBlock);
  const int c0 = (int)cta_of(blk * t.ntiles, t.units, p.ctas), c1 = (int)cta_of((blk + 1) * t.ntiles - 1, t.units, p.ctas);
  float best = -1e30f, sec = -1e30f;
  int grp = INT_MAX;
  bool good = true;
  auto join = [&](float b, float s, int gi) {
    sec = fmaxf(fmaxf(sec, s), fminf(best, b));
    grp = b > best ? gi : b < best ? grp : min(grp, gi);
    best = fmaxf(best, b);
  };
  for (int i = lane; i < kParts * (c1 - c0 + 1); i += 32) {
    const float* q = t.part + ((size_t)(c0 + i / kParts + blk) * kParts + i % kParts) * 3 * kBlock + r;
    join(q[0], q[kBlock], __float_as_int(q[2 * kBlock]));
    good = good && t.status[c0 + i / kParts] == 1u;
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    const float b = __shfl_xor_sync(0xFFFFFFFFu, best, d), s = __shfl_xor_sync(0xFFFFFFFFu, sec, d);
    join(b, s, __shfl_xor_sync(0xFFFFFFFFu, grp, d));
  }
  good = __all_sync(0xFFFFFFFFu, good);
  // another group within T of the best and no label wanted: not a fold, whatever the group holds (95 % of
  // 3x3x3's ids); scores are whole numbers
  if (good && !p.aux && !p.gap && sec + 10.f * p.C >= 0.f && best - sec < (float)p.T) {
    if (lane == 0) p.phen[row] = -1;
    return;
  }
  int M = 0, second = -1, first = 0;  // best score, second best (< 0: none), lowest minimiser
  if (good) {
    const int c = kGroup * grp + lane;
    const int x = (unsigned)c < (unsigned)p.S_dir ? exact_score(p.rec + (size_t)c * p.rec_words, p.NE, e, o) : -1;
    M = (int)best + 10 * p.C;
    const uint32_t eq = __ballot_sync(0xFFFFFFFFu, x == M);
    first = kGroup * grp + __ffs(eq) - 1;
    second = __popc(eq) > 1 ? M : max(__reduce_max_sync(0xFFFFFFFFu, x == M ? -1 : x), (int)fmaxf(sec, -1e6f) + 10 * p.C);
    good = eq != 0u;
  }
  if (!good) {
    // a wait gave up in one of the runs: the sequence is scored against every conformation here
    if (p.err && lane == 0) atomicOr(p.err, 1u);
    int b = -1, s = -1, f = INT_MAX;
    for (int c = lane; c < p.S_dir; c += 32) {
      const int x = exact_score(p.rec + (size_t)c * p.rec_words, p.NE, e, o);
      if (x > b) {
        s = b;
        b = x;
        f = c;
      } else {
        s = max(s, x);
      }
    }
    M = __reduce_max_sync(0xFFFFFFFFu, b);
    first = __reduce_min_sync(0xFFFFFFFFu, b == M ? f : INT_MAX);
    second = __popc(__ballot_sync(0xFFFFFFFFu, b == M)) > 1 ? M : __reduce_max_sync(0xFFFFFFFFu, b == M ? s : b);
  }
  if (lane == 0) {
    int gap = second < 0 ? INT_MAX : M - second;
    if (p.prune) gap = min(gap, p.T);
    const int cls = __ldg(p.conf_class + first);
    p.phen[row] = gap >= p.T ? cls : -1;
    if (p.aux) p.aux[row] = cls;
    if (p.gap) p.gap[row] = gap;
  }
}

// The pairs in contact in some conformation, and the conformations' 0/1 rows over them in slab order.  A
// table above kMaxTable is never built (tc_nk -1); one that finds no room now is tried again by the next
// call (tc_nk stays 0), and this call's ids go to the caller's other kernel.
int scan_tc_tables(const hp_structs* cs, hp::DevTables** out) {
  hp::DevTables* dt = nullptr;
  const int rc = hp::device_tables(cs, &dt);
  if (rc != HP_OK) return rc;
  hp_structs* s = const_cast<hp_structs*>(cs);
  std::lock_guard<std::mutex> lock(s->mu);
  *out = dt;
  if (dt->tc_nk != 0) return HP_OK;
  std::vector<int> col((size_t)hp::kMaxHalf * hp::kMaxHalf, -1);
  const uint8_t* ct = s->contacts.data();
  const size_t nc = (size_t)s->S_dir * s->C;
  auto pair_of = [&](size_t c) {
    const int i = ct[2 * c], j = ct[2 * c + 1];
    return (i & 1) ? (j / 2) * hp::kMaxHalf + i / 2 : (i / 2) * hp::kMaxHalf + j / 2;
  };
  for (size_t c = 0; c < nc; c++) col[pair_of(c)] = 0;
  std::vector<uint16_t> pairs;
  for (size_t v = 0; v < col.size(); v++)
    if (col[v] == 0) {
      col[v] = (int)pairs.size();
      pairs.push_back((uint16_t)((v / hp::kMaxHalf) | ((v % hp::kMaxHalf) << 8)));
    }
  const int cpad = (int)pairs.size();  // the constant column
  const int nk = (cpad + 1 + 31) / 32, ntiles = (s->S_dir + kTile - 1) / kTile;
  pairs.resize((size_t)32 * nk, 0x1F1F);  // bit 31 of both halves is clear: the constant -10
  const size_t bytes = (size_t)ntiles * nk * kSlabB;
  if (bytes > kMaxTable) {
    dt->tc_nk = -1;
    return HP_OK;
  }
  // the device's memory first: a call that gets none leaves tc_nk at 0 and costs no more than this
  uint8_t* d_tab = nullptr;
  uint16_t* d_pairs = nullptr;
  hp::TableUpload up;
  up.alloc(reinterpret_cast<void**>(&d_tab), bytes);
  const cudaError_t got = up.alloc(reinterpret_cast<void**>(&d_pairs), pairs.size() * 2);
  const std::unique_ptr<uint8_t[]> tab(got == cudaSuccess ? new (std::nothrow) uint8_t[bytes]() : nullptr);
  if (!tab) {
    cudaFree(d_tab);
    cudaFree(d_pairs);
    cudaGetLastError();
    return HP_OK;
  }
  auto at = [&](size_t conf, int k) -> uint8_t& {
    const size_t t = conf / kTile, r = conf % kTile;
    return tab[(t * nk + k / 32) * kSlabB + (r / 8) * 256 + ((k / 16) & 1) * 128 + (r % 8) * 16 + k % 16];
  };
  for (size_t c = 0; c < nc; c++) at(c / s->C, col[pair_of(c)]) = (uint8_t)kF1;
  for (size_t c = (size_t)s->S_dir; c < (size_t)ntiles * kTile; c++) at(c, cpad) = (uint8_t)kF448;
  up.copy(d_tab, tab.get(), bytes);
  up.copy(d_pairs, pairs.data(), pairs.size() * 2);
  if (up.finish() != cudaSuccess) {
    cudaFree(d_tab);
    cudaFree(d_pairs);
    cudaGetLastError();
    return HP_OK;
  }
  dt->tc_tab = d_tab;
  dt->tc_pairs = d_pairs;
  dt->tc_nk = nk;
  dt->tc_ntiles = ntiles;
  return HP_OK;
}

// Stream-ordered scratch from a pool of the library's own, which keeps one launch's worth (kPoolKeep) when the
// streams are idle.  The device's default pool gives its memory back at every synchronisation, and the call
// after it waits for new mappings: one id of 5x5 and a synchronisation took 220 us so (59 on the warp
// scan) and 40 from this pool, 16,384 ids of 4x5 228 and 46 (70).  Freed with the library.
cudaError_t pool_scratch(hp_structs* s, hp::DevTables* dt, size_t bytes, cudaStream_t st, char** out) {
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(s->mu);
    if (!dt->scan_pool) {
      hp::TableUpload relaxed;
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dt->device;
      unsigned long long keep = kPoolKeep;
      cudaError_t e = cudaMemPoolCreate(&pool, &props);
      if (e != cudaSuccess) return e;
      e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return e;
      }
      dt->scan_pool = pool;
    }
    pool = dt->scan_pool;
  }
  return cudaMallocFromPoolAsync(reinterpret_cast<void**>(out), bytes, pool, st);
}

struct ScratchLease {
  std::shared_ptr<hp::GraphScratch> pool;
  size_t block;
};

void CUDART_CB end_lease(void* p) {  // (may run on a thread of the driver: no CUDA calls)
  ScratchLease* l = static_cast<ScratchLease*>(p);
  {
    std::lock_guard<std::mutex> lock(l->pool->mu);
    if (l->block < l->pool->blocks.size()) l->pool->blocks[l->block].used = false;  // (empty: the library is gone)
  }
  delete l;
}

// Scratch for a scan that is being captured into graph; NULL where there is none.  Stream-ordered memory would
// put memory nodes into the graph, of which only one instance may then exist and which no other graph
// may hold; this block is the graph's by reference instead (a user object, which its instances and
// clones hold too).
char* graph_scratch(hp_structs* s, hp::DevTables* dt, cudaGraph_t graph, size_t bytes) try {
  {
    std::lock_guard<std::mutex> lock(s->mu);
    if (!dt->graph_scratch) dt->graph_scratch = std::make_shared<hp::GraphScratch>();
  }
  // no CUDA call is made under the pool's lock, which end_lease takes
  hp::GraphScratch& pool = *dt->graph_scratch;
  std::unique_ptr<ScratchLease> lease(new ScratchLease{dt->graph_scratch, 0});
  void* p = nullptr;
  {
    std::lock_guard<std::mutex> lock(pool.mu);
    std::vector<hp::GraphScratch::Block>& b = pool.blocks;
    size_t best = b.size();  // the smallest free block that is large enough, or else a place without memory
    for (size_t i = 0; i < b.size(); i++)
      if (!b[i].used && b[i].bytes >= bytes && (best == b.size() || b[i].bytes < b[best].bytes)) best = i;
    for (size_t i = 0; i < b.size() && best == b.size(); i++)
      if (!b[i].used && !b[i].p) best = i;
    if (best == b.size()) b.push_back({nullptr, 0, false});
    b[best].used = true;
    p = b[best].p;
    lease->block = best;
  }
  bool ok = p != nullptr;
  if (!ok) {
    hp::TableUpload relaxed;
    ok = relaxed.alloc(&p, bytes) == cudaSuccess;
    std::lock_guard<std::mutex> lock(pool.mu);
    pool.blocks[lease->block].p = ok ? p : nullptr;
    pool.blocks[lease->block].bytes = ok ? bytes : 0;
  }
  cudaUserObject_t obj = nullptr;
  ok = ok && cudaUserObjectCreate(&obj, lease.get(), end_lease, 1, cudaUserObjectNoDestructorSync) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    end_lease(lease.release());
    return nullptr;
  }
  lease.release();  // now the object's
  if (cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove) != cudaSuccess) {
    cudaGetLastError();
    cudaUserObjectRelease(obj, 1);
    return nullptr;
  }
  return static_cast<char*>(p);
} catch (const std::bad_alloc&) {
  return nullptr;
}

}  // namespace

namespace hp {

// *done = 0: the caller's other kernel has to take the ids (the table or the scratch does not fit).
int scan_tc(const hp_structs* s, const ScanTc& a, cudaStream_t st, long long* done) {
  *done = 0;
  DevTables* dt = nullptr;
  int rc = scan_tc_tables(s, &dt);
  if (rc != HP_OK) return rc;
  if (dt->tc_nk <= 0) return HP_OK;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  TcParams p{};
  p.tab = dt->tc_tab;
  p.pairs = dt->tc_pairs;
  p.nk = dt->tc_nk;
  p.ntiles = dt->tc_ntiles;
  const int abytes = 2 * p.nk * kSlabA;
  // The largest stage (slabs per wait, copy and commit) that leaves one stage beside the tile's, which
  // stay resident for both halves.  Every stage costs the issuers a wait and a commit: 65,536 ids of
  // 6x6 (10 slabs) took 925 us with stages of 2 slabs, 812 with 3 and 700 with 5; 3x3x3 (5 slabs)
  // 1464 us with 1, 878 with 3 and 627 with 5 (before other changes: 648 and 573 us now).
  for (p.cs = std::min(p.nk, kMaxStage); p.cs >= 1; p.cs--) {
    p.nslots = std::min(kMaxSlots, (kSmemMax - 128 - abytes) / (p.cs * kSlabB));
    if (p.nslots > (p.nk + p.cs - 1) / p.cs) break;
  }
  if (p.cs < 1) return HP_OK;
  p.spin = (uint32_t)std::min<long long>(wait_limit(kSpin), 0xFFFFFFFFll);
  const size_t smem = (size_t)abytes + (size_t)p.nslots * p.cs * kSlabB + 128;
  cudaError_t e = cudaFuncSetAttribute(scan_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(scan_tc_kernel)");
  const long long chunk = std::min<long long>(a.n, kChunk);
  const long long blocks = (chunk + kBlock - 1) / kBlock;
  const size_t part = sizeof(float) * 3 * kParts * kBlock * (size_t)(blocks + sms);
  const size_t bytes = (part + sizeof(unsigned) * sms + 255) / 256 * 256;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaGraph_t graph = nullptr;
  if (cudaStreamGetCaptureInfo(st, &capture, nullptr, &graph) != cudaSuccess) cudaGetLastError();
  const bool captured = capture == cudaStreamCaptureStatusActive;
  char* scratch = nullptr;
  if (captured) {  // each launch its own part: instances of the graph may run side by side
    scratch = graph_scratch(const_cast<hp_structs*>(s), dt, graph, bytes * (size_t)((a.n + chunk - 1) / chunk));
  } else if (pool_scratch(const_cast<hp_structs*>(s), dt, bytes, st, &scratch) != cudaSuccess) {
    cudaGetLastError();
    scratch = nullptr;
  }
  if (!scratch) return HP_OK;
  p.part = reinterpret_cast<float*>(scratch);
  p.status = reinterpret_cast<unsigned*>(scratch + part);
  for (long long off = 0; off < a.n && rc == HP_OK; off += chunk) {
    p.n = std::min(chunk, a.n - off);
    p.ids = a.ids ? a.ids + off : nullptr;
    p.base = a.base + (unsigned long long)off;
    p.units = (p.n + kBlock - 1) / kBlock * p.ntiles;
    const int ctas = (int)std::min<long long>(sms, p.units);
    scan_tc_kernel<<<ctas, kThreads, smem, st>>>(p);
    ResolveParams r{};
    r.t = p;
    r.ctas = ctas;
    r.rec = dt->rec;
    r.conf_class = dt->conf_class;
    r.rec_words = s->rec_words;
    r.NE = s->NE;
    r.C = s->C;
    r.S_dir = s->S_dir;
    r.T = a.T;
    r.prune = a.prune;
    r.phen = a.phen + off;
    r.aux = a.aux ? a.aux + off : nullptr;
    r.gap = a.gap ? a.gap + off : nullptr;
    r.counters = reinterpret_cast<unsigned long long*>(a.counters);
    r.err = a.err;
    scan_tc_resolve<<<(unsigned)((p.n + 7) / 8), 256, 0, st>>>(r);
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(e, "tensor-core scan: launch");
    if (captured) {
      p.part = reinterpret_cast<float*>(reinterpret_cast<char*>(p.part) + bytes);
      p.status = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(p.status) + bytes);
    }
  }
  if (!captured) cudaFreeAsync(scratch, st);
  if (rc == HP_OK) *done = a.n;
  return rc;
}

}  // namespace hp
