// The full matrix of Eq. 2 numerators (Section 2.3 of arXiv 2008.05612): for every ordered pair of
// phenotypes (q, p), the number of single flips from a genotype of q to a genotype of p,
//   M[q][p] = #{(g, i) : P(g) = q, P(g xor 2^i) = p},  phi_pq = M[q][p] / (N N_q),
// with index S standing for the deleterious phenotype -1.  The matrix is sparse (a phenotype's
// neighbours are few: 0.86% of the 3x3x3 phenotypes touch the top fold, Section 3.2), so it is
// returned in compressed rows with columns ascending.
//
// Where the counts come from.  The diagonal M[p][p] and the -1 column M[p][S] are the robustness
// numerators; flips are symmetric (g -> h is a flip iff h -> g is), so the -1 row is the -1 column
// transposed, M[S][p] = M[p][S].  Only the flips between two different non-deleterious phenotypes (4%
// of the 3x3x3 neighbours) need a table, a hash table keyed by (q, p), which the robustness passes fill
// beside their own counters: they have every folding genotype and its flips in shared memory already.
//
// From the table to sorted rows: count the rows' entries, one scan gives the row offsets, scatter the
// entries into their rows, and sort each row on its own (a row has about 20 entries): a warp ranks
// each entry among its row's by comparison; a row of more than kWarpRow entries is ranked by a bitmap
// of its columns (at most 65,536 bits) in shared memory.  The -1 column is always a row's last entry, and
// the -1 row's entries follow from a scan over the phenotypes.  Nothing waits for the host until the end.
// The map of 2^25 ids at the 3x3x3 folding density (0.9 million entries) took 5.41 ms with a second pass
// over the map for the table and a bitonic sort of all entries (210 launches); now 0.63 ms, of which the
// passes over the map are 0.40.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "hp_internal.h"

namespace {

constexpr unsigned kErrRange = 4u;   // a map entry outside [-1, S)
constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr int kWarpRow = 256;        // longest row that one warp sorts
constexpr int kScanThreads = 1024;

struct Phi {
  hp::PhiTable table;
  const unsigned long long *neutral, *to_del;  // S + 1 each
  uint32_t *rowcnt, *cursor;   // per row: table entries; where its next entry goes
  uint32_t *delrank;           // phenotypes below p with a flip to -1
  uint32_t *big, *nbig;        // rows longer than kWarpRow
  int32_t* scol;               // entries by row, unsorted
  unsigned long long* scnt;
  unsigned long long cap;
  unsigned long long* nnz;
  const unsigned* err;
  int S;
  unsigned long long* at;      // S + 2 row offsets
  unsigned long long* row_ptr; // the caller's
  int32_t* col;
  unsigned long long* count;
};

// the call fails: nothing may be written (the buffers hold cap entries)
__device__ __forceinline__ bool failed(const Phi& p) { return *p.err != 0u || *p.nnz > p.cap; }

__global__ void phi_count_rows(const Phi p) {
  const unsigned long long cap = 1ull << p.table.log2cap, stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride) {
    const uint32_t k = p.table.keys[s];
    if (k != kEmpty) atomicAdd(&p.rowcnt[k >> 16], 1u);
  }
}

// A row's entries (low 40 bits): the table's, the diagonal and the -1 column; and its -1 flip (high 24 bits).
__device__ __forceinline__ unsigned long long row_size(const Phi& p, int q) {
  const unsigned long long del = p.to_del[q] != 0;
  return (unsigned long long)p.rowcnt[q] + (p.neutral[q] != 0) + del + (del << 40);
}

// Sum of v over the CTA's threads before this one; *total over all of them.
__device__ unsigned long long scan_block(unsigned long long v, unsigned long long* part, unsigned long long* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += y;
  }
  __syncthreads();  // part may still be read by a previous scan
  if (lane == 31) part[warp] = incl;
  __syncthreads();
  unsigned long long before = 0, all = 0;
  for (int w = 0; w < kScanThreads / 32; w++) {
    const unsigned long long x = part[w];
    if (w < warp) before += x;
    all += x;
  }
  *total = all;
  return before + incl - v;
}

// Row offsets, a CTA per 1,024 rows.  Each CTA adds up the rows before its own itself (coalesced, at most
// 65,534 rows: 3x3x3's 51,704 took one CTA with a run of rows per thread 197 us).  Row S has an entry per
// phenotype with a flip to -1, and its diagonal.
__global__ void __launch_bounds__(kScanThreads) phi_scan_rows(const Phi p) {
  __shared__ unsigned long long part[kScanThreads / 32];
  constexpr unsigned long long kLow = (1ull << 40) - 1;
  const int q0 = blockIdx.x * kScanThreads, q = q0 + threadIdx.x;
  unsigned long long sum = 0, base, mine;
#pragma unroll 4
  for (int i = threadIdx.x; i < q0; i += kScanThreads) sum += row_size(p, i);
  scan_block(sum, part, &base);
  const unsigned long long v = q < p.S ? row_size(p, q) : 0ull;
  const unsigned long long at = base + scan_block(v, part, &mine);
  if (q < p.S) {
    p.at[q] = at & kLow;
    p.cursor[q] = (uint32_t)(at & kLow);
    p.delrank[q] = (uint32_t)(at >> 40);
  }
  if (q == p.S) {
    p.at[q] = at & kLow;
    *p.nnz = p.at[q + 1] = (at & kLow) + (at >> 40) + (p.neutral[q] != 0);
  }
}

__global__ void phi_scatter(const Phi p) {
  if (failed(p)) return;
  const unsigned long long cap = 1ull << p.table.log2cap, stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride) {
    const uint32_t k = p.table.keys[s];
    if (k == kEmpty) continue;
    const uint32_t at = atomicAdd(&p.cursor[k >> 16], 1u);
    p.scol[at] = (int32_t)(k & 0xFFFFu);
    p.scnt[at] = p.table.counts[s];
  }
}

// One warp per row: rank the table's entries and the diagonal among themselves, append the -1 column,
// write this phenotype's entry of the -1 row, and copy the row's offset out.
__global__ void phi_sort_rows(const Phi p) {
  if (failed(p)) return;
  const int q = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (q > p.S) return;
  if (lane == 0) p.row_ptr[q] = p.at[q];
  if (q == p.S) {
    if (lane == 0) p.row_ptr[q + 1] = p.at[q + 1];
    if (lane == 0 && p.neutral[q]) {
      const unsigned long long at = p.at[q + 1] - 1;
      p.col[at] = q;
      p.count[at] = p.neutral[q];
    }
    return;
  }
  const unsigned long long beg = p.at[q];
  const int n = (int)p.rowcnt[q];
  const unsigned long long diag = p.neutral[q], del = p.to_del[q];
  if (n > kWarpRow) {
    if (lane == 0) p.big[atomicAdd(p.nbig, 1u)] = (uint32_t)q;
  } else {
    int below = 0;  // entries left of the diagonal
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      const int32_t c = i < n ? p.scol[beg + i] : INT32_MAX;
      int rank = c > q && diag ? 1 : 0;
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int32_t other = j0 + lane < n ? p.scol[beg + j0 + lane] : INT32_MAX;
#pragma unroll 8
        for (int j = 0; j < 32; j++) rank += __shfl_sync(0xFFFFFFFFu, other, j) < c;
      }
      below += __popc(__ballot_sync(0xFFFFFFFFu, c < q));
      if (i < n) {
        p.col[beg + rank] = c;
        p.count[beg + rank] = p.scnt[beg + i];
      }
    }
    if (lane == 0 && diag) {
      p.col[beg + below] = q;
      p.count[beg + below] = diag;
    }
  }
  if (lane == 0 && del) {
    const unsigned long long last = p.at[q + 1] - 1, at = p.at[p.S] + p.delrank[q];
    p.col[last] = p.S;
    p.count[last] = del;
    p.col[at] = q;
    p.count[at] = del;
  }
}

// The long rows, one per CTA at a time: a bitmap of the row's columns and the prefix sums of its words.
__global__ void __launch_bounds__(kScanThreads) phi_sort_big_rows(const Phi p) {
  if (failed(p)) return;
  constexpr int kWords = 2048;  // 65,536 columns
  __shared__ uint32_t bits[kWords], pre[kWords];
  __shared__ unsigned long long part[kScanThreads / 32];
  for (uint32_t r = blockIdx.x; r < *p.nbig; r += gridDim.x) {
    const int q = (int)p.big[r];
    const unsigned long long beg = p.at[q];
    const int n = (int)p.rowcnt[q];
    const unsigned long long diag = p.neutral[q];
    for (int w = threadIdx.x; w < kWords; w += kScanThreads) bits[w] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kScanThreads) {
      const uint32_t c = (uint32_t)p.scol[beg + i];
      atomicOr(&bits[c >> 5], 1u << (c & 31));
    }
    if (threadIdx.x == 0 && diag) atomicOr(&bits[q >> 5], 1u << (q & 31));
    __syncthreads();
    const uint32_t w0 = __popc(bits[2 * threadIdx.x]), w1 = __popc(bits[2 * threadIdx.x + 1]);
    unsigned long long total;
    const uint32_t before = (uint32_t)scan_block(w0 + w1, part, &total);
    pre[2 * threadIdx.x] = before;
    pre[2 * threadIdx.x + 1] = before + w0;
    __syncthreads();
    auto rank = [&](uint32_t c) { return pre[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u)); };
    for (int i = threadIdx.x; i < n; i += kScanThreads) {
      const uint32_t c = (uint32_t)p.scol[beg + i];
      p.col[beg + rank(c)] = (int32_t)c;
      p.count[beg + rank(c)] = p.scnt[beg + i];
    }
    if (threadIdx.x == 0 && diag) {
      p.col[beg + rank((uint32_t)q)] = q;
      p.count[beg + rank((uint32_t)q)] = diag;
    }
    __syncthreads();  // the bitmap is cleared for the next row
  }
}

int sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

}  // namespace

extern "C" int hp_phi_matrix(const int32_t* d_phen, int32_t N, int32_t S, uint64_t cap, uint64_t* d_row_ptr,
                             int32_t* d_col, uint64_t* d_count, uint64_t* h_nnz, void* stream) {
  if (!d_phen || !d_row_ptr || !d_col || !d_count || !h_nnz) return hp::fail(HP_EINVAL, "hp_phi_matrix: NULL pointer");
  if (N < 1 || N > 40) return hp::fail(HP_EINVAL, "hp_phi_matrix: N must be in [1, 40]");
  if (S < 1 || S >= 0xFFFF) return hp::fail(HP_EINVAL, "hp_phi_matrix: S must be in [1, 65534]");
  if (cap < 1 || cap > (1ull << 30)) return hp::fail(HP_EINVAL, "hp_phi_matrix: cap must be in [1, 2^30]");
  cudaStream_t st = (cudaStream_t)stream;
  *h_nnz = 0;
  // hash table: twice the off-diagonal capacity, a power of two (at least 2^10)
  int log2cap = 10;
  while ((1ull << log2cap) < 2 * cap && log2cap < 31) log2cap++;
  const unsigned long long hcap = 1ull << log2cap;
  // scratch: [err 8][nnz 8][negcount 8][nbig 8][neutral (S+1)][to_del (S+1)][rowcnt S] | cursor, delrank, big (S
  // each), row offsets (S + 2) | counts | entry counts | entry columns | keys; the first part and the counts start at zero
  const size_t rows = ((size_t)S + 1) / 2 * 2 + 2;  // 32-bit words per row array, 8-byte multiples
  const size_t head = 32 + 16ull * (size_t)(S + 1) + 4 * rows;
  const size_t tail = 3 * 4 * rows + 8 * ((size_t)S + 2);
  const size_t bytes = head + tail + hcap * 8 + cap * 8 + (cap + 1) / 2 * 8 + hcap * 4;
  char* scratch = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&scratch), bytes, st);
  if (e != cudaSuccess) return hp::cuda_fail(e, "hp_phi_matrix: cudaMallocAsync");
  unsigned* err = reinterpret_cast<unsigned*>(scratch);
  unsigned long long* negcount = reinterpret_cast<unsigned long long*>(scratch + 16);
  unsigned long long* neutral = reinterpret_cast<unsigned long long*>(scratch + 32);
  unsigned long long* to_del = neutral + (S + 1);
  Phi p;
  p.neutral = neutral;
  p.to_del = to_del;
  p.rowcnt = reinterpret_cast<uint32_t*>(to_del + (S + 1));
  p.cursor = p.rowcnt + rows;
  p.delrank = p.cursor + rows;
  p.big = p.delrank + rows;
  p.nbig = reinterpret_cast<uint32_t*>(scratch + 24);
  p.at = reinterpret_cast<unsigned long long*>(p.big + rows);
  p.table.counts = reinterpret_cast<unsigned long long*>(scratch + head + tail);
  p.table.log2cap = log2cap;
  p.scnt = p.table.counts + hcap;
  p.scol = reinterpret_cast<int32_t*>(p.scnt + cap);
  p.table.keys = reinterpret_cast<uint32_t*>(p.scol + (cap + 1) / 2 * 2);
  p.cap = cap;
  p.nnz = reinterpret_cast<unsigned long long*>(scratch + 8);
  p.err = err;
  p.S = S;
  p.row_ptr = reinterpret_cast<unsigned long long*>(d_row_ptr);
  p.col = d_col;
  p.count = reinterpret_cast<unsigned long long*>(d_count);
  int rc = HP_OK;
  e = cudaMemsetAsync(scratch, 0, head + tail + hcap * 8, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p.table.keys, 0xFF, hcap * 4, st);
  if (e == cudaSuccess) e = hp::launch_robustness(d_phen, N, S, neutral, to_del, negcount, err, st, &p.table);
  if (e == cudaSuccess) {
    const unsigned grid = (unsigned)std::min<unsigned long long>((hcap + 255) / 256, (unsigned long long)sms() * 16);
    phi_count_rows<<<grid, 256, 0, st>>>(p);
    phi_scan_rows<<<S / kScanThreads + 1, kScanThreads, 0, st>>>(p);
    phi_scatter<<<grid, 256, 0, st>>>(p);
    phi_sort_rows<<<(S + 1 + 7) / 8, 256, 0, st>>>(p);
    phi_sort_big_rows<<<sms(), kScanThreads, 0, st>>>(p);
    e = cudaGetLastError();
  }
  unsigned long long head_words[2] = {0, 0};  // error word, entries
  if (e == cudaSuccess) e = cudaMemcpyAsync(head_words, scratch, 16, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) rc = hp::cuda_fail(e, "hp_phi_matrix: counting");
  const unsigned herr = (unsigned)head_words[0];
  const unsigned long long nnz = head_words[1];
  if (rc == HP_OK && (herr & kErrRange)) rc = hp::fail(HP_EINVAL, "hp_phi_matrix: map entry outside [-1, S)");
  if (rc == HP_OK && ((herr & hp::kErrPhiFull) || nnz > cap)) {
    *h_nnz = (herr & hp::kErrPhiFull) ? 0 : nnz;
    rc = hp::fail(HP_ENOMEM, "hp_phi_matrix: the matrix has more than cap = " + std::to_string(cap) +
                                 " nonzero entries; call again with cap >= *h_nnz (0: unknown, at least 2 x cap)");
  }
  if (rc == HP_OK) *h_nnz = nnz;
  cudaFreeAsync(scratch, st);
  return rc;
}
