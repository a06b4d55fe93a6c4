// decompress_kernels.cu - the round trip (§4.1: ROIs restored exactly over the
// up-sampled background) and the ROI mask.
//
//   parse (header, layout, decoding tables) -> decode (chunk-parallel
//   canonical Huffman) -> lorenzo outliers -> row prefix sums -> column prefix
//   sums + dequantisation -> prequantisation outliers -> up-sampling -> ROI
//   windows and status (k_dec_roi_coded and k_dec_windows, roi_coder.cu)
//
// Every index taken from the stream is bounds-checked; a failed check marks
// the frame ROIBIN_ERR_CORRUPT_STREAM and skips the access.
#include <cuda_runtime.h>

#include <algorithm>

#include "roibin_internal.cuh"

namespace roibin {

constexpr int32_t kSentinel = INT32_MIN;  // delta of a code-0 bin until its outlier arrives
constexpr uint32_t kDecSparseMax = 1024;  // other symbols per chunk at most, for a sparse frame

__device__ __forceinline__ void mark_corrupt(Scratch& s, uint32_t f) {
  s.status[f] = ROIBIN_ERR_CORRUPT_STREAM;
}

// The fields of a stream's header (24 words), checked against the context's
// geometry and each other as the oracle checks them; the stream's layout.
__device__ bool read_header(const uint32_t* hdr, const DevParams& p, uint64_t base, uint64_t in_bytes, DecInfo& di) {
  di = DecInfo{};
  di.base = base;
  const uint32_t roi_h = hdr[5] & 0xFFFFu, roi_w = hdr[5] >> 16;
  const uint32_t bh = hdr[6] & 0xFFFFu, bw = hdr[6] >> 16;
  di.eb = __uint_as_float(hdr[7]);
  di.two_eb = __fmul_rn(2.0f, di.eb);
  di.R = (int32_t)hdr[8];
  di.roi_h = (int32_t)roi_h;
  di.roi_w = (int32_t)roi_w;
  di.nsym = 2u * hdr[8];
  FramePlan& pl = di.pl;
  di.roi_coding = hdr[19];
  di.roi_bytes = hdr[20];
  di.roi_words = hdr[21];
  di.back_ref = hdr[22];
  pl.n_peaks = hdr[9];
  pl.n_lo = hdr[10];
  pl.n_pq = hdr[11];
  pl.n_words = hdr[15];
  const uint64_t total = (uint64_t)hdr[16] | ((uint64_t)hdr[17] << 32);
  bool ok = !(hdr[0] != kMagic || hdr[1] != kVersion || hdr[2] != p.P || hdr[3] != p.H || hdr[4] != p.W ||
              bh != (uint32_t)p.bh || bw != (uint32_t)p.bw || roi_h < 1 || roi_h > 63 || roi_w < 1 ||
              roi_w > 63 || hdr[8] < 2 || hdr[8] > 512 || hdr[12] != p.M || hdr[13] != kChunk ||
              hdr[14] != p.n_chunks || pl.n_lo > p.M || pl.n_pq > p.M || pl.n_words > p.M ||
              pl.n_peaks > 65535u || !(di.eb > 0.0f) || !isfinite(di.two_eb) ||
              hdr[18] != (p.dims == 2 ? 0u : (uint32_t)p.dims) ||  // the context's Lorenzo dimension
              di.roi_coding > 2 || (di.roi_coding == 0 && (di.roi_bytes | di.roi_words) != 0) ||
              di.back_ref > 63);  // a chunk holds at most 64 frames
  pl.off_peaks = kHeaderBytes;
  pl.off_roi = pl.off_peaks + align16((uint64_t)pl.n_peaks * 6);
  pl.off_len = pl.off_roi + (di.roi_coding == 0 ? align16((uint64_t)pl.n_peaks * roi_h * roi_w * 4) : 0);
  pl.off_cidx = pl.off_len + (di.back_ref == 0 ? align16(di.nsym) : 0);  // lengths: a chunk's head only
  pl.off_lo = pl.off_cidx + align16((uint64_t)p.n_chunks * 4);
  pl.off_pq = pl.off_lo + align16((uint64_t)pl.n_lo * 8);
  pl.off_bits = pl.off_pq + align16((uint64_t)pl.n_pq * 8);
  pl.total = pl.off_bits + align16((uint64_t)pl.n_words * 4);
  di.off_roi_sec = pl.total;  // the ROI section after the bitstream (roi coding 1, 2)
  pl.total += di.roi_bytes;
  if (pl.total != total || base + pl.total > in_bytes) ok = false;
  return ok;
}

// [2][P] first entry of each panel in the frame's Lorenzo and prequantisation
// outlier lists (in the compressor's outlier slots, free while decompressing: two
// words a panel at least).
__device__ __forceinline__ uint32_t* dec_list_starts(const Scratch& s, const DevParams& p, uint32_t f) {
  return s.pq_mask + (size_t)f * 2 * p.P;
}

// parse: one block per frame.  Reads the header and the code lengths (its own,
// or those of its chunk's head, back_ref frames earlier in the call), builds
// the canonical decoding tables and the prefix table, checks that both outlier
// lists are strictly ascending and inside the frame, and records where each
// panel's outliers start in them.
__global__ void __launch_bounds__(256) k_dec_parse(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  __shared__ uint32_t hdr[24], hhdr[24];
  __shared__ int ok;
  __shared__ uint64_t len_at;  // byte offset of the code lengths in the input
  __shared__ uint32_t cnt[34], first[34], idx0[34];
  __shared__ __align__(4) uint8_t lens[kMaxSymbols];
  __shared__ uint16_t order[kMaxSymbols];
  __shared__ uint32_t nsym_s;
  __shared__ int sparse;
  const uint32_t f = blockIdx.x;
  DecInfo di = {};
  if (threadIdx.x == 0) {
    s.dec_zero[f] = 0;
    s.thr_count[f] = 0;  // blocks of k_dec_windows done with the frame
    ok = 1;
    const uint64_t base = a.offsets[f];
    if ((base & 15u) != 0 || base + kHeaderBytes > a.in_bytes) ok = 0;
    if (ok) {
      const uint32_t* h = reinterpret_cast<const uint32_t*>(a.in + base);
      for (int i = 0; i < 24; ++i) hdr[i] = h[i];
      ok = read_header(hdr, p, base, a.in_bytes, di) ? 1 : 0;
      len_at = base + di.pl.off_len;
    }
    // a stream without code lengths takes its chunk head's: the frame back_ref
    // earlier in this call, which must be a valid stream keeping its own
    // lengths, with the same alphabet
    if (ok && di.back_ref != 0) {
      DecInfo hd;
      const uint64_t hb = di.back_ref <= f ? a.offsets[f - di.back_ref] : 0;
      ok = di.back_ref <= f && (hb & 15u) == 0 && hb + kHeaderBytes <= a.in_bytes;
      if (ok) {
        const uint32_t* h = reinterpret_cast<const uint32_t*>(a.in + hb);
        for (int i = 0; i < 24; ++i) hhdr[i] = h[i];
        ok = read_header(hhdr, p, hb, a.in_bytes, hd) && hd.back_ref == 0 && hd.R == di.R;
        len_at = hb + hd.pl.off_len;
      }
    }
    if (!ok) {
      s.status[f] = ROIBIN_ERR_CORRUPT_STREAM;
      s.dec_info[f] = di;
    }
  }
  __syncthreads();
  if (!ok) return;
  if (threadIdx.x != 0) read_header(hdr, p, a.offsets[f], a.in_bytes, di);  // every thread's copy
  __syncthreads();
  // canonical decoding tables: count per length, first code per length, index
  // of the first symbol of each length in the (length, symbol) order.
  const uint8_t* base = a.in + di.base;
  uint32_t* tab = s.dec_table + (size_t)f * kDecTableWords;
  if (threadIdx.x < 34) cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) nsym_s = di.nsym;
  __syncthreads();
  for (uint32_t k = threadIdx.x; k < di.nsym; k += blockDim.x) {
    const uint32_t L = a.in[len_at + k];
    lens[k] = (uint8_t)L;
    if (L > 32) ok = 0;
    else if (L > 0) atomicAdd(&cnt[L], 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t c = 0;
    uint32_t prev = 0, idx = 0;
    uint64_t kraft = 0;  // sum of 2^(32 - L): a complete code sums to 2^32
    first[0] = idx0[0] = 0;
    for (uint32_t L = 1; L <= 32; ++L) {
      first[L] = 0;
      idx0[L] = idx;
      if (cnt[L]) {
        c = prev == 0 ? 0 : (c + cnt[prev]) << (L - prev);
        first[L] = (uint32_t)c;
        prev = L;
        kraft += (uint64_t)cnt[L] << (32 - L);
      }
      idx += cnt[L];
    }
    // a code with one symbol of length 1 is allowed (kraft = 2^31)
    const bool single = idx == 1 && cnt[1] == 1;
    if (idx == 0 || (kraft != (1ull << 32) && !single)) ok = 0;
    sparse = cnt[1] != 0;
  }
  __syncthreads();
  // sparse frame: with a length-1 code every other code takes 2 bits or more,
  // so a chunk of n symbols in w words holds at most 32 w - n other symbols
  if (sparse) {
    const uint32_t* cidx = reinterpret_cast<const uint32_t*>(base + di.pl.off_cidx);
    for (uint32_t k = threadIdx.x; k < p.n_chunks; k += blockDim.x) {
      const uint32_t w0 = cidx[k], w1 = k + 1 < p.n_chunks ? cidx[k + 1] : di.pl.n_words;
      const uint32_t n = min(p.M, k * kChunk + kChunk) - k * kChunk;
      if (w1 < w0 || 32ull * (w1 - w0) > (uint64_t)n + kDecSparseMax) sparse = 0;
    }
  }
  if (threadIdx.x <= 32) {
    const uint32_t L = threadIdx.x;
    tab[L] = L ? cnt[L] : 0;
    tab[34 + L] = first[L];
    tab[68 + L] = idx0[L];
  }
  // symbols in (length, symbol) order: rank among same-length smaller symbols
  for (uint32_t k = threadIdx.x; k < nsym_s; k += blockDim.x) {
    const uint32_t L = lens[k];
    if (L == 0 || L > 32) continue;
    const uint32_t same = L * 0x01010101u;  // four lengths a word
    uint32_t rank = 0;
    for (uint32_t j = 0; j + 4 <= k; j += 4)
      rank += __popc(__vcmpeq4(*reinterpret_cast<const uint32_t*>(lens + j), same)) >> 3;
    for (uint32_t j = k & ~3u; j < k; ++j) rank += lens[j] == L;
    tab[102 + idx0[L] + rank] = k;
    order[idx0[L] + rank] = (uint16_t)k;
  }
  __syncthreads();
  // prefix table.  Canonical codes grow with their length: entry e starts with a
  // code of at most L bits when it is below end[L], the first 12-bit value past
  // those codes, so its code's length is 1 + the ends it has reached.
  if (ok) {
    uint32_t end[kDecLutBits + 1];
    end[0] = 0;
#pragma unroll
    for (uint32_t L = 1; L <= kDecLutBits; ++L) end[L] = cnt[L] ? (first[L] + cnt[L]) << (kDecLutBits - L) : end[L - 1];
    for (uint32_t w = threadIdx.x; w < kDecLutWords; w += blockDim.x) {
      uint32_t word = 0;
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        const uint32_t e = 2 * w + h;
        uint32_t L = 1;
#pragma unroll
        for (uint32_t l = 1; l <= kDecLutBits; ++l) L += e >= end[l];
        if (L <= kDecLutBits) word |= ((L << 10) | order[idx0[L] + (e >> (kDecLutBits - L)) - first[L]]) << (16 * h);
      }
      tab[kDecCanonWords + w] = word;
    }
  }
  // outlier lists: strictly ascending bin indices below M; the first entry of
  // each panel's run goes to the panel's start slot
  const uint32_t Mp = p.Hb * p.Wb;
  for (int list = 0; list < 2; ++list) {
    const uint2* v = reinterpret_cast<const uint2*>(base + (list == 0 ? di.pl.off_lo : di.pl.off_pq));
    const uint32_t n = list == 0 ? di.pl.n_lo : di.pl.n_pq;
    uint32_t* start = dec_list_starts(s, p, f) + (list == 0 ? 0 : p.P);
    if (n == 0)
      for (uint32_t q = threadIdx.x; q < p.P; q += blockDim.x) start[q] = 0;
    for (uint32_t e = threadIdx.x; e < n; e += blockDim.x) {
      const uint32_t x = v[e].x;
      const uint32_t px = e ? v[e - 1].x : 0u;
      if (x >= p.M || (e > 0 && px >= x)) {
        ok = 0;
        continue;
      }
      const uint32_t q1 = x / Mp;
      for (uint32_t q = e ? px / Mp + 1 : 0; q <= q1; ++q) start[q] = e;
      if (e == n - 1)
        for (uint32_t q = q1 + 1; q < p.P; ++q) start[q] = n;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!ok) s.status[f] = ROIBIN_ERR_CORRUPT_STREAM;
    else s.status[f] = ROIBIN_OK;
    di.sparse = sparse ? 1u : 0u;
    s.dec_info[f] = di;
  }
}

// lorenzo: scatter the Lorenzo-outlier deltas (must land on code-0 bins, in
// strictly ascending order).
__global__ void k_dec_lorenzo(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const DecInfo& di = s.dec_info[f];
  if (blockIdx.x == 0 && threadIdx.x == 0 && s.dec_zero[f] != di.pl.n_lo) mark_corrupt(s, f);
  const uint2* lo = reinterpret_cast<const uint2*>(a.in + di.base + di.pl.off_lo);
  int32_t* dq = s.dq + (size_t)f * p.M;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < di.pl.n_lo; e += gridDim.x * blockDim.x) {
    const uint2 v = lo[e];
    const bool ordered = e == 0 || lo[e - 1].x < v.x;
    if (v.x >= p.M || !ordered || dq[v.x] != kSentinel) {
      mark_corrupt(s, f);
      continue;
    }
    dq[v.x] = (int32_t)v.y;
  }
}

// rows: inclusive prefix sum along each binned row (one warp per row).
__global__ void k_dec_rows(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const uint32_t row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= p.P * p.Hb) return;
  uint32_t* r = reinterpret_cast<uint32_t*>(s.dq + (size_t)f * p.M + (size_t)row * p.Wb);
  uint32_t carry = 0;  // unsigned: wraps instead of overflowing on corrupt input
  for (uint32_t j0 = 0; j0 < p.Wb; j0 += 32) {
    const uint32_t j = j0 + lane_id();
    const uint32_t v = j < p.Wb ? r[j] : 0u;
    const uint32_t inc = warp_incl_scan(v) + carry;
    if (j < p.Wb) r[j] = inc;
    carry = __shfl_sync(0xffffffffu, inc, 31);
  }
}

// cols: prefix sum down each column of a binned panel, then b^ = fl(q * 2eb)
// (dequant), or the sums back in place for the 3-D inverse (k_dec_stack_out).
__global__ void k_dec_cols(DevParams p, Scratch s, DecArgs a, int dequant) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.P * p.Wb) return;
  const uint32_t pn = t / p.Wb, j = t - pn * p.Wb;
  const float two_eb = s.dec_info[f].two_eb;
  uint32_t* dq = reinterpret_cast<uint32_t*>(s.dq + (size_t)f * p.M + (size_t)pn * p.Hb * p.Wb);
  float* bh = s.bhat + (size_t)f * p.M + (size_t)pn * p.Hb * p.Wb;
  uint32_t q = 0;
  for (uint32_t i = 0; i < p.Hb; ++i) {
    q += dq[(size_t)i * p.Wb + j];
    if (dequant) bh[(size_t)i * p.Wb + j] = __fmul_rn((float)(int32_t)q, two_eb);
    else dq[(size_t)i * p.Wb + j] = q;
  }
}

// stack (3-D inverse, last axis): prefix sum across the panels at each binned
// position of their 2-D sums, b^ = fl(q * 2eb) and the bin's pixels.  The three
// axes' prefix sums commute, so rows, columns, then panels inverts the 3-D
// predictor.  kVec: bin 2 x 2, W % 4 == 0, 16-byte aligned frames: a thread takes
// two bins and stores a float4 on each of their rows; else a thread takes a pixel
// column of a binned row.  Four panels' sums are read ahead.  HBM-bound: the sums
// in and the pixels out, once each; with k_dec_panel<true> it replaces a pass
// each over the int32 sums for rows, columns, panels and up-sampling: 40 CSPAD-like
// frames 226 -> 125 us.
template <bool kVec>
__global__ void __launch_bounds__(256) k_dec_stack_out(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, cols = kVec ? p.W / 4 : p.W;
  const uint32_t i = t / cols, c = t - i * cols;
  if (i >= p.Hb) return;
  const float two_eb = s.dec_info[f].two_eb;
  const uint32_t plane = p.Hb * p.Wb;
  const uint32_t* dq = reinterpret_cast<const uint32_t*>(s.dq) + (size_t)f * p.M + (size_t)i * p.Wb;
  const uint32_t r0 = i * p.bh, r1 = min(p.H, r0 + p.bh);
  float* out = a.out + (size_t)f * p.frame_px + (size_t)r0 * p.W;
  uint32_t q0 = 0, q1 = 0;
  constexpr uint32_t U = 4;
  for (uint32_t p0 = 0; p0 < p.P; p0 += U) {
    uint2 v[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      v[u] = make_uint2(0u, 0u);
      if (p0 + u < p.P) {
        const uint32_t* at = dq + (size_t)(p0 + u) * plane;
        if (kVec) v[u] = __ldcs(reinterpret_cast<const uint2*>(at) + c);
        else v[u].x = __ldg(at + c / p.bw);
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      if (p0 + u >= p.P) break;
      q0 += v[u].x;
      q1 += v[u].y;
      const float b0 = __fmul_rn((float)(int32_t)q0, two_eb), b1 = __fmul_rn((float)(int32_t)q1, two_eb);
      float* px = out + (size_t)(p0 + u) * p.H * p.W;
      for (uint32_t r = r0; r < r1; ++r, px += p.W) {
        if (kVec) __stcs(reinterpret_cast<float4*>(px) + c, make_float4(b0, b0, b1, b1));
        else __stcs(px + c, b0);
      }
    }
  }
}

// The prequantisation outliers' pixels, over those of k_dec_stack_out (the lists
// were checked by the parse step).
__global__ void k_dec_pq_pixels(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const DecInfo& di = s.dec_info[f];
  const uint2* pq = reinterpret_cast<const uint2*>(a.in + di.base + di.pl.off_pq);
  const uint32_t plane = p.Hb * p.Wb;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < di.pl.n_pq; e += gridDim.x * blockDim.x) {
    const uint2 v = pq[e];
    const uint32_t pn = v.x / plane, b = v.x - pn * plane, i = b / p.Wb, j = b - i * p.Wb;
    const uint32_t r1 = min(p.H, (i + 1) * p.bh), c1 = min(p.W, (j + 1) * p.bw);
    float* panel = a.out + (size_t)f * p.frame_px + (size_t)pn * p.H * p.W;
    for (uint32_t r = i * p.bh; r < r1; ++r)
      for (uint32_t c = j * p.bw; c < c1; ++c) panel[(size_t)r * p.W + c] = __uint_as_float(v.y);
  }
}

// chain (1-D inverse): after the row sums, every binned row adds the sum of
// all rows before it in the frame's row-major order.  One block per frame
// walks the rows in tiles of blockDim.x, scanning the tile's row totals.
constexpr uint32_t kChainThreads = 1024;
__global__ void __launch_bounds__(kChainThreads) k_dec_chain(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  __shared__ uint32_t carry[kChainThreads];
  __shared__ uint32_t warp_sum[kChainThreads / 32];
  const uint32_t f = blockIdx.x;
  if (s.status[f] != ROIBIN_OK) return;
  const float two_eb = s.dec_info[f].two_eb;
  const uint32_t* dq = reinterpret_cast<const uint32_t*>(s.dq + (size_t)f * p.M);
  float* bh = s.bhat + (size_t)f * p.M;
  const uint32_t rows = p.P * p.Hb, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  uint32_t base = 0;  // sum of every row before the tile (unsigned: wraps like the stream's int32)
  for (uint32_t r0 = 0; r0 < rows; r0 += kChainThreads) {
    const uint32_t r = r0 + tid;
    const uint32_t total = r < rows ? dq[(size_t)r * p.Wb + p.Wb - 1] : 0u;  // the row's inclusive sum
    const uint32_t inc = warp_incl_scan(total);
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = warp_incl_scan(warp_sum[lane]);
      warp_sum[lane] = w;
    }
    __syncthreads();
    carry[tid] = base + (warp ? warp_sum[warp - 1] : 0u) + inc - total;  // exclusive
    const uint32_t tile_sum = warp_sum[31];
    __syncthreads();
    const uint32_t n = min(kChainThreads, rows - r0);
    for (uint32_t k = warp; k < n; k += kChainThreads / 32) {
      const size_t row = (size_t)(r0 + k) * p.Wb;
      const uint32_t c = carry[k];
      for (uint32_t j = lane; j < p.Wb; j += 32)
        bh[row + j] = __fmul_rn((float)(int32_t)(dq[row + j] + c), two_eb);
    }
    base += tile_sum;
    __syncthreads();
  }
}

// pq: prequantisation outliers overwrite b^ with their stored bits.
__global__ void k_dec_pq(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const DecInfo& di = s.dec_info[f];
  const uint2* pq = reinterpret_cast<const uint2*>(a.in + di.base + di.pl.off_pq);
  float* bh = s.bhat + (size_t)f * p.M;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < di.pl.n_pq; e += gridDim.x * blockDim.x) {
    const uint2 v = pq[e];
    const bool ordered = e == 0 || pq[e - 1].x < v.x;
    if (v.x >= p.M || !ordered) {
      mark_corrupt(s, f);
      continue;
    }
    bh[v.x] = __uint_as_float(v.y);
  }
}

// upsample: every pixel takes its bin's value.
__global__ void k_dec_upsample(DevParams p, Scratch s, DecArgs a, int vec4) {
  chain_wait();
  const uint32_t f = blockIdx.y;
  if (s.status[f] != ROIBIN_OK) return;
  const float* bh = s.bhat + (size_t)f * p.M;
  float* out = a.out + (size_t)f * p.frame_px;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  if (vec4) {  // bin 2 x 2, W % 4 == 0: 4 pixels = 2 bins
    const uint64_t n4 = p.frame_px / 4;
    const uint32_t W4 = p.W / 4;
    for (uint64_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += stride) {
      const uint32_t rowg = (uint32_t)(e / W4), c4 = (uint32_t)(e - (uint64_t)rowg * W4);
      const uint32_t pn = rowg / p.H, r = rowg - pn * p.H;
      const float2 v = *reinterpret_cast<const float2*>(bh + ((size_t)pn * p.Hb + r / 2) * p.Wb + 2 * c4);
      reinterpret_cast<float4*>(out)[e] = make_float4(v.x, v.x, v.y, v.y);
    }
    return;
  }
  for (uint64_t e = blockIdx.x * blockDim.x + threadIdx.x; e < p.frame_px; e += stride) {
    const uint32_t rowg = (uint32_t)(e / p.W), c = (uint32_t)(e - (uint64_t)rowg * p.W);
    const uint32_t pn = rowg / p.H, r = rowg - pn * p.H;
    out[e] = bh[((size_t)pn * p.Hb + r / p.bh) * p.Wb + c / p.bw];
  }
}

// ---------------------------------------------------------------------------
// The decoders of both paths: several lanes per 4,096-symbol chunk.
//
// A Huffman code resynchronises: a decoder started inside a codeword meets the
// true codeword boundaries again after a few codewords.  So the chunk's bits
// are cut into equal ranges, one per lane.  Every lane decodes its range from
// the range's first bit, counting codewords, and says where the first codeword
// past its range starts.  A lane whose left neighbour says another start than
// the one it used decodes again from there, until no start changes (lane 0's is
// right from the outset, so at most 31 times; once on detector frames).  Then
// the starts are the serial decoder's own, an exclusive scan of the counts gives
// every lane the index of its first symbol, and a last pass decodes and stores.
// Bits of the zero padding may decode as symbols past the chunk's last one; they
// are not stored.
//
// A thread per chunk (4,096 dependent lookups) kept too few lanes busy: a
// 60-frame epix10k batch has 7,920 chunks.  What bounds these is the chain of
// window, lookup and advance per lane, three times over.  us, a thread per
// chunk -> now: 60 epix10k frames (2.9 bits a symbol, dense) 1,460 -> 187; one
// CSPAD-like frame (1.02 bits, sparse) 54 -> 9.5, 400 of them 90 -> 44 (within calls; 57
// with caches flushed); 40 of them as residuals for the multi-pass path 943 -> 66.
//
// Two shortcuts, as the code allows:
//   - When a code of length 1 exists it is the all-zero code, so a run of z zero
//     bits is z copies of its symbol, taken in one step (count of leading zeros).
//   - Other codes: the next 12 bits index a table (several codewords at once in
//     the dense decoder; codes of more than 12 bits are found by their length).
//
// What is stored:
//   k_dec_dense<true> (the multi-pass path): every symbol's residual, as int32, at
//   its bin;
//   k_dec_sparse: a frame the parse step marked sparse (a length-1 code, and each chunk's
//   bit count leaves room for at most kDecSparseMax other symbols) stores only
//   each chunk's other symbols (dec_list): the panel kernel fills the rest, so the
//   frame's symbols never go through device memory;
//   k_dec_dense<false>: every symbol of the other frames, in the
//   [n][n_chunks * kChunk] u16 symbol array.
// Dense symbols are collected in shared memory (the lanes' runs start 128
// symbols apart, so a word of padding per 32 keeps them off one bank) and leave
// in whole lines.
constexpr uint32_t kDecWarps = 8;              // warps per block
constexpr uint32_t kDecStageWords = 704;       // a chunk's words in shared memory (longer chunks: through L1)
constexpr uint32_t kDecSymWords = kChunk / 2 + kChunk / 64;  // its symbols, padded
constexpr uint32_t kDecWarpWords = kDecStageWords + 8 + kDecSymWords;
constexpr uint32_t kDecLutSize = 1u << kDecLutBits;
// the canonical tables, the pair table, the count table, the warps' words and symbols: 2 blocks per SM
constexpr uint32_t kDecPairAt = kDecCanonWords, kDecCountAt = kDecPairAt + kDecLutSize,
                   kDecLongAt = kDecCountAt + kDecLutSize / 4, kDecWarpAt = kDecLongAt + 40;
constexpr uint32_t kDecSmem = (kDecWarpAt + kDecWarps * kDecWarpWords) * 4;
static_assert(2 * (kDecSmem + 1024) <= 228 * 1024, "two dense decoder blocks share an SM");
static_assert(kDecWarps * kDecWarpWords >= kDecLutWords, "the prefix table is read from the warps' area");

// A code of more than kDecLutBits bits from the top of `win` (the next 32 bits):
// its length, 0 when no code matches; the symbol in `sym`.
__device__ __noinline__ uint32_t decode_long(const uint32_t* tab, uint32_t win, uint32_t& sym) {
  for (uint32_t L = kDecLutBits + 1; L <= 32; ++L) {
    const uint32_t n = tab[L], d = (win >> (32 - L)) - tab[34 + L];
    if (d < n) {  // a code below the first of its length wraps far above n
      sym = tab[102 + tab[68 + L] + d];
      return L;
    }
  }
  return 0;
}

// A sparse frame's symbols, as the decoder leaves them for the panel kernel:
// chunk k lists its symbols other than the length-1 code's, in order, as
// (position in the chunk << 16) | symbol, in the first half of the chunk's slot
// of the symbol array; the count per chunk goes to the [n][n_chunks] array the
// compressor uses for its per-chunk outlier offsets (free while decompressing).
__device__ __forceinline__ uint32_t* dec_list(const Scratch& s, const DevParams& p, uint32_t f, uint32_t k) {
  return reinterpret_cast<uint32_t*>(s.codes + ((size_t)f * p.n_chunks + k) * kChunk);
}
__device__ __forceinline__ uint32_t* dec_list_count(const Scratch& s, const DevParams& p, uint32_t f) {
  return s.chunk_lo + (size_t)f * p.n_chunks;
}
static_assert(kDecSparseMax * 4 <= kChunk * 2, "a chunk's list fits its slot of the symbol array");

// Decodes the codewords of a chunk that start in bits [at, limit), at most
// `room` of them; `word(i)` is the chunk's word i (0 past its end).  `other(i,
// sym)` is called for the i-th codeword of the range unless it belongs to a run
// of the length-1 code; sym is 0xFFFFFFFF where no code matches (one bit is
// skipped then).  Returns the codewords decoded; `at` becomes the bit after them.
// The window is fetched anew for every codeword (two words, one funnel shift):
// fewer instructions than a bit buffer with its refills.
template <class Word, class Other>
__device__ __forceinline__ uint32_t decode_range(const uint32_t* tab, const uint16_t* lut, uint32_t& at, uint32_t limit,
                                                 uint32_t room, Word word, Other other) {
  uint32_t pos = at, n = 0;
  while (pos < limit && n < room) {
    const uint32_t win = __funnelshift_l(word((pos >> 5) + 1), word(pos >> 5), pos & 31u);
    if ((int32_t)win >= 0) {  // a run of the length-1 code
      const uint32_t z = min((uint32_t)__clz(win), min(limit - pos, room - n));
      n += z;
      pos += z;
    } else {
      const uint32_t ent = lut[win >> (32 - kDecLutBits)];
      uint32_t sym = ent & 1023u, L = ent >> 10;
      if (L == 0) L = decode_long(tab, win, sym);
      if (L == 0) {
        L = 1;
        sym = 0xFFFFFFFFu;
      }
      other(n, sym);
      ++n;
      pos += L;
    }
  }
  at = pos;
  return n;
}

// The lanes' starts and counts of one chunk of nw words, decoded by a warp (lane l
// covers bits [l nw, (l + 1) nw)).  `n`: codewords of the lane's range; `listed`: those not in
// runs; `start`: the bit its first codeword starts at; `end`: the bit after its last.
// `note(j, i, sym)` sees the j-th listed codeword, the range's i-th; what a lane's
// last pass noted stands.
template <class Decode, class Note>
__device__ __forceinline__ void sync_ranges(uint32_t nw, uint32_t& start, uint32_t& end, uint32_t& n,
                                            uint32_t& listed, Decode decode, Note note) {
  const uint32_t lane = lane_id(), limit = (lane + 1) * nw;
  start = end = lane * nw;
  listed = 0;
  n = decode(end, limit, 0xFFFFFFFFu, [&](uint32_t i, uint32_t sym) { note(listed++, i, sym); });
  for (uint32_t round = 0; round < 32; ++round) {
    const uint32_t left = __shfl_up_sync(0xffffffffu, end, 1);
    const bool again = lane > 0 && left != start;
    if (!__any_sync(0xffffffffu, again)) break;
    if (again) {
      start = end = left;
      listed = 0;
      n = decode(end, limit, 0xFFFFFFFFu, [&](uint32_t i, uint32_t sym) { note(listed++, i, sym); });
    }
  }
}

// Loads the frame's decoding tables; false when the frame is not sparse (or not OK).
// Other blocks of the frame may mark it corrupt meanwhile, so the decision is read once
// and shared.
__device__ __forceinline__ bool dec_load_tables(const Scratch& s, uint32_t f, uint32_t* tab, int* go) {
  if (threadIdx.x == 0) *go = s.status[f] == ROIBIN_OK && s.dec_info[f].sparse != 0;
  __syncthreads();
  if (!*go) return false;
  const uint4* src = reinterpret_cast<const uint4*>(s.dec_table + (size_t)f * kDecTableWords);
  static_assert(kDecTableWords % 4 == 0, "table copied in 16-byte pieces");
  for (uint32_t i = threadIdx.x; i < kDecTableWords / 4; i += blockDim.x) reinterpret_cast<uint4*>(tab)[i] = src[i];
  __syncthreads();
  return true;
}

// Sparse frames: a warp per chunk, words read through L1, a few chunks per warp
// (each block loads the frame's tables once).  A lane notes the first kDecNotes
// listed codewords of its range while it settles, so that most lanes (a CSPAD-like
// frame's list about one in two) write their list without decoding the range again:
// 1,000 frames 157 -> 125 us, 200 frames 43 -> 35 us.
constexpr uint32_t kDecNotes = 8;
__global__ void __launch_bounds__(kDecWarps * 32) k_dec_sparse(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  __shared__ __align__(16) uint32_t tab[kDecTableWords];
  __shared__ uint32_t notes[kDecNotes * kDecWarps * 32];
  __shared__ int go;
  const uint32_t f = blockIdx.y, lane = lane_id();
  if (!dec_load_tables(s, f, tab, &go)) return;
  const uint16_t* lut = reinterpret_cast<const uint16_t*>(tab + kDecCanonWords);
  const DecInfo& di = s.dec_info[f];
  const uint8_t* base = a.in + di.base;
  const uint32_t n_words = di.pl.n_words;
  const uint32_t* cidx = reinterpret_cast<const uint32_t*>(base + di.pl.off_cidx);
  const uint32_t zsym = tab[102];  // the length-1 code is code 0: first in the (length, symbol) order
  for (uint32_t k = blockIdx.x * kDecWarps + (threadIdx.x >> 5); k < p.n_chunks; k += gridDim.x * kDecWarps) {
    const uint32_t w0 = cidx[k], w1 = k + 1 < p.n_chunks ? cidx[k + 1] : n_words;
    const uint32_t n_sym = min(p.M, k * kChunk + kChunk) - k * kChunk;
    // a chunk of n symbols takes at most n words
    bool bad = w0 > w1 || w1 > n_words || w1 - w0 > kChunk;
    const uint32_t nw = bad ? 0u : w1 - w0;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(base + di.pl.off_bits) + w0;
    auto decode = [&](uint32_t& at, uint32_t limit, uint32_t room, auto other) {
      return decode_range(tab, lut, at, limit, room, [&](uint32_t i) { return i < nw ? __ldg(words + i) : 0u; }, other);
    };
    uint32_t start, end, n, listed;
    uint32_t* noted = notes + threadIdx.x;  // position in the range << 16 | symbol; a range is at most 4,127 bits
    sync_ranges(nw, start, end, n, listed, decode, [&](uint32_t j, uint32_t i, uint32_t sym) {
      if (j < kDecNotes) noted[j * (kDecWarps * 32)] = i << 16 | (sym & 0xFFFFu);
    });
    uint32_t first = warp_incl_scan(n), at_list = warp_incl_scan(listed);
    if (lane == 31 && first < n_sym) bad = true;  // the chunk's bits end too early
    first -= n;
    at_list -= listed;
    uint32_t zeros = 0, wrote = 0;
    if (!bad && first < n_sym && n > 0) {
      uint32_t* list = dec_list(s, p, f, k);
      const uint32_t room = min(n, n_sym - first);
      // the noted codewords stand for the range when they are all of its listed ones, each a
      // code, and inside the chunk: what the range holds past the chunk's end is then runs of
      // the length-1 code, a bit each
      bool all = listed <= kDecNotes;
      for (uint32_t j = 0; all && j < listed; ++j) {
        const uint32_t v = noted[j * (kDecWarps * 32)];
        all = (v >> 16) < room && (v & 0xFFFFu) != 0xFFFFu;
      }
      uint32_t bit = start;
      if (all) {
        for (; wrote < listed; ++wrote) {
          const uint32_t v = noted[wrote * (kDecWarps * 32)];
          if (at_list + wrote >= kDecSparseMax) bad = true;
          else list[at_list + wrote] = v + (first << 16);
          zeros += (v & 0xFFFFu) == 0;
        }
        bit = end - (n - room);
      } else {
        decode(bit, (lane + 1) * nw, room, [&](uint32_t i, uint32_t sym) {
          if (sym > 0xFFFFu || at_list + wrote >= kDecSparseMax) bad = true;
          else list[at_list + wrote] = ((first + i) << 16) | sym;
          ++wrote;
          zeros += sym == 0;
        });
      }
      if (zsym == 0) zeros += room - wrote;
      // the chunk's last symbol: its words must end with it
      if (first + room == n_sym && (bit + 31) / 32 != nw) bad = true;
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    zeros = __reduce_add_sync(0xffffffffu, zeros);
    wrote = __reduce_add_sync(0xffffffffu, wrote);
    if (lane == 0) {
      dec_list_count(s, p, f)[k] = any_bad ? 0u : wrote;
      if (any_bad) mark_corrupt(s, f);
      if (zeros) atomicAdd(s.dec_zero + f, zeros);
    }
  }
}

// The dense decoder's tables in shared memory, from the frame's prefix table:
//   pair[x], x the next 12 bits: bits 0-9 the first symbol, 20-23 its length (0:
//     longer than 12 bits); bits 10-19 the second, 24-27 the length of both (0:
//     the second does not end inside the 12 bits);
//   count[x]: bits 0-3 the codewords that end inside the 12 bits, 4-7 their length.
// The counting passes then take about four codewords of an epix10k frame per
// lookup and the storing pass two.
__device__ __forceinline__ void build_dense_tables(const uint32_t* frame_tab, uint32_t* sm) {
  uint16_t* lut = reinterpret_cast<uint16_t*>(sm + kDecWarpAt);
  for (uint32_t i = threadIdx.x; i < kDecCanonWords; i += blockDim.x) sm[i] = frame_tab[i];
  for (uint32_t i = threadIdx.x; i < kDecLutWords; i += blockDim.x) sm[kDecWarpAt + i] = frame_tab[kDecCanonWords + i];
  __syncthreads();
  uint8_t* count = reinterpret_cast<uint8_t*>(sm + kDecCountAt);
  const uint32_t most = sm[1] ? 2u : kDecLutBits;  // with a length-1 code the runs are taken by counting zeros
  for (uint32_t x = threadIdx.x; x < kDecLutSize; x += blockDim.x) {
    uint32_t pair = 0, at = 0, n = 0;
    for (;;) {
      const uint32_t ent = lut[(x << at) & (kDecLutSize - 1)], L = ent >> 10;
      if (L == 0 || at + L > kDecLutBits) break;
      at += L;
      if (n == 0) pair = (ent & 1023u) | (L << 20);
      if (n == 1) pair |= ((ent & 1023u) << 10) | (at << 24);
      if (++n == most) break;
    }
    sm[kDecPairAt + x] = pair;
    count[x] = (uint8_t)(n | (at << 4));
  }
  // codes of 13 .. 32 bits: the last 32-bit window that starts with a code of at
  // most L bits (canonical codes grow with their length), then where the symbols
  // of length L start, less its first code
  if (threadIdx.x < 20) {
    const uint32_t L = kDecLutBits + 1 + threadIdx.x;
    uint32_t m = L;
    while (m > 1 && sm[m] == 0) --m;
    sm[kDecLongAt + threadIdx.x] = (uint32_t)(((uint64_t)sm[34 + m] + sm[m]) << (32 - m)) - 1u;
    sm[kDecLongAt + 20 + threadIdx.x] = 102 + sm[68 + L] - sm[34 + L];
  }
  __syncthreads();
}

// A code of more than kDecLutBits bits from the top of `win`, by those tables:
// the lengths 13 .. 20 are compared at once.
__device__ __forceinline__ uint32_t decode_long_fast(const uint32_t* sm, uint32_t win, uint32_t& sym) {
  const uint4* last = reinterpret_cast<const uint4*>(sm + kDecLongAt);
  const uint4 a = last[0], b = last[1];
  uint32_t i = (win > a.x) + (win > a.y) + (win > a.z) + (win > a.w) + (win > b.x) + (win > b.y) + (win > b.z) + (win > b.w);
  if (i == 8) {
    while (i < 20 && win > sm[kDecLongAt + i]) ++i;
    if (i == 20) return 0;
  }
  const uint32_t L = kDecLutBits + 1 + i;
  sym = sm[sm[kDecLongAt + 20 + i] + (win >> (32 - L))];
  return L;
}

// Every symbol: a warp per chunk.  kDeltas: every frame, its residuals at their
// bins; else the frames that are not sparse, their symbols.
template <bool kDeltas>
__global__ void __launch_bounds__(kDecWarps * 32, 2) k_dec_dense(DevParams p, Scratch s, DecArgs a) {
  chain_wait();
  extern __shared__ __align__(16) uint32_t dec_sm[];
  __shared__ int go;
  const uint32_t f = blockIdx.y, lane = lane_id(), warp = threadIdx.x >> 5;
  // other blocks of the frame may mark it corrupt meanwhile: read once and shared
  if (threadIdx.x == 0) go = s.status[f] == ROIBIN_OK && (kDeltas || s.dec_info[f].sparse == 0);
  __syncthreads();
  if (!go) return;
  build_dense_tables(s.dec_table + (size_t)f * kDecTableWords, dec_sm);
  const uint32_t* tab = dec_sm;
  const uint32_t* pair = dec_sm + kDecPairAt;
  const uint8_t* counts = reinterpret_cast<const uint8_t*>(dec_sm + kDecCountAt);
  uint32_t* stage = dec_sm + kDecWarpAt + warp * kDecWarpWords;
  uint32_t* symw = stage + kDecStageWords + 8;
  uint16_t* syms = reinterpret_cast<uint16_t*>(symw);
  auto slot = [](uint32_t i) { return i + 2 * (i >> 6); };  // u16 index of symbol i in syms
  const DecInfo& di = s.dec_info[f];
  const uint8_t* base = a.in + di.base;
  const uint32_t n_words = di.pl.n_words;
  const uint32_t* cidx = reinterpret_cast<const uint32_t*>(base + di.pl.off_cidx);
  const bool zrun = tab[1] != 0;  // the length-1 code is code 0: its symbol comes first in the (length, symbol) order
  const uint32_t zsym = tab[102];
  for (uint32_t k = blockIdx.x * kDecWarps + warp; k < p.n_chunks; k += gridDim.x * kDecWarps) {
    const uint32_t w0 = cidx[k], w1 = k + 1 < p.n_chunks ? cidx[k + 1] : n_words;
    const uint32_t nw = w1 - w0, n_sym = min(p.M, k * kChunk + kChunk) - k * kChunk;
    if (w0 > w1 || w1 > n_words || nw > kChunk) {  // a chunk of n symbols takes at most n words
      if (lane == 0) mark_corrupt(s, f);
      continue;
    }
    const uint32_t* words = reinterpret_cast<const uint32_t*>(base + di.pl.off_bits) + w0;
    const bool staged = nw <= kDecStageWords;
    if (staged) {
      for (uint32_t i = lane; i < nw; i += 32) stage[i] = words[i];
      if (lane < 8) stage[nw + lane] = 0;  // read past the end: a window starts below bit 32 nw
    }
    if (zrun)
      for (uint32_t i = lane; i < kDecSymWords; i += 32) symw[i] = zsym * 0x10001u;
    __syncwarp();
    auto window = [&](uint32_t pos) {  // the 32 bits from bit pos < 32 nw
      const uint32_t i = pos >> 5;
      const uint32_t hi = staged ? stage[i] : __ldg(words + i);
      const uint32_t lo = staged ? stage[i + 1] : (i + 1 < nw ? __ldg(words + i + 1) : 0u);
      return __funnelshift_l(lo, hi, pos & 31u);
    };
    // counting pass over the codewords that start in [at, limit)
    auto count_range = [&](uint32_t& at, uint32_t limit, uint32_t, auto) {
      uint32_t pos = at, n = 0;
      while (pos < limit) {
        const uint32_t win = window(pos);
        if (zrun && (int32_t)win >= 0) {
          const uint32_t z = min((uint32_t)__clz(win), limit - pos);
          n += z;
          pos += z;
          continue;
        }
        const uint32_t c = counts[win >> (32 - kDecLutBits)];
        if (c != 0 && pos + kDecLutBits <= limit) {
          n += c & 15u;
          pos += c >> 4;
          continue;
        }
        uint32_t L = (pair[win >> (32 - kDecLutBits)] >> 20) & 15u, sym;
        if (L == 0) L = max(1u, decode_long_fast(dec_sm, win, sym));
        ++n;
        pos += L;
      }
      at = pos;
      return n;
    };
    const uint32_t limit = (lane + 1) * nw;
    uint32_t start, end, n, listed;
    sync_ranges(nw, start, end, n, listed, count_range, [](uint32_t, uint32_t, uint32_t) {});
    const uint32_t first = warp_incl_scan(n) - n;
    // the storing pass: this lane's codewords are symbols first .. first + n - 1
    uint32_t zeros = 0;
    bool bad = false;
    if (first < n_sym && n > 0) {
      const uint32_t room = min(n, n_sym - first);
      uint32_t pos = start, i = 0;
      while (i < room) {
        const uint32_t win = window(pos);
        if (zrun && (int32_t)win >= 0) {  // prefilled
          const uint32_t z = min((uint32_t)__clz(win), room - i);
          if (zsym == 0) zeros += z;
          i += z;
          pos += z;
          continue;
        }
        const uint32_t e = pair[win >> (32 - kDecLutBits)];
        uint32_t L = (e >> 20) & 15u, sym = e & 1023u;
        if (L == 0) {
          L = decode_long_fast(dec_sm, win, sym);
          if (L == 0) {
            bad = true;
            break;
          }
        }
        syms[slot(first + i)] = (uint16_t)sym;
        zeros += sym == 0;
        ++i;
        if ((e >> 24) != 0 && i < room) {
          const uint32_t sym2 = (e >> 10) & 1023u;
          syms[slot(first + i)] = (uint16_t)sym2;
          zeros += sym2 == 0;
          ++i;
          L = e >> 24;
        }
        pos += L;
      }
      // the chunk's last symbol: its words must end with it
      if (first + room == n_sym && (pos + 31) / 32 != nw) bad = true;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, first + n, 31);
    bad = __any_sync(0xffffffffu, bad) || total < n_sym;
    for (int d = 16; d > 0; d >>= 1) zeros += __shfl_xor_sync(0xffffffffu, zeros, d);
    if (lane == 0) {
      if (bad) mark_corrupt(s, f);
      if (zeros) atomicAdd(s.dec_zero + f, zeros);
    }
    if (bad) continue;
    __syncwarp();
    if constexpr (kDeltas) {
      int32_t* dq = s.dq + (size_t)f * p.M + (size_t)k * kChunk;
      for (uint32_t i = lane; i < n_sym; i += 32) {
        const uint32_t u = syms[slot(i)];
        dq[i] = u ? (int32_t)u - di.R : kSentinel;
      }
    } else {
      uint32_t* out = reinterpret_cast<uint32_t*>(s.codes + ((size_t)f * p.n_chunks + k) * kChunk);
      for (uint32_t i = lane; 2 * i < n_sym; i += 32) out[i] = symw[i + (i >> 5)];  // a slot holds the whole last word
    }
    __syncwarp();  // the warp's area is free for its next chunk
  }
}

// Places the outliers of one strip.  The run of the list that belongs to the
// panel is ascending, so the strip's entries are the first ones still unplaced:
// thread t takes entry cur + t, and the count of threads that found theirs in
// the strip advances the cursor for everyone.  `place(bin, value)` returns false
// on a corrupt entry.
template <class F>
__device__ __forceinline__ uint32_t place_strip_outliers(const uint2* v, uint32_t cur, uint32_t end, uint32_t sb1,
                                                         F place, bool& bad) {
  for (;;) {
    const uint32_t e = cur + threadIdx.x;
    bool in = false;
    if (e < end) {
      const uint2 x = v[e];
      in = x.x < sb1;
      if (in && !place(x.x, x.y)) bad = true;
    }
    const uint32_t n_in = (uint32_t)__syncthreads_count(in);
    cur += n_in;
    if (n_in < blockDim.x) return cur;
  }
}

// The panel path: k_dec_sparse and k_dec_dense, then one block per (panel, frame).  Strip by strip (sb binned rows):
//   symbols -> deltas in shared memory (code 0: sentinel), Lorenzo outliers in;
//   column prefix sums carried from the strip above (thread per column);
//   row prefix sums, b^ = fl(q * 2eb) and the row's pixels by a warp per row from
//   registers (bin width 2).  Strips with prequantisation outliers and other bin
//   widths take them apart: a thread per row segment, b^ back to the tile, the
//   outliers in, then the output rows.  The one pass instead of three took the
//   kernel from 185 to 108 us on 60 epix10k frames and from 650 to 617 us on 400
//   CSPAD-like frames (5.96 TB/s of pixels written, 0.88 of the copy rate).
// k_dec_roi_coded or k_dec_windows then overwrites the pixels of the ROI windows.
// The 2-D prefix sum wraps modulo 2^32 in any order, so column-then-row equals
// the row-then-column definition.
// kSums (3-D predictor): the panel's 2-D sums go to s.dq instead of pixels;
// k_dec_stack_out adds them up across the panels and writes the pixels.
// The symbols of the next strip arrive by a 1-D TMA bulk copy (a 16-byte
// aligned superset of the strip) while the block works on the current one.
constexpr int kPanelThreads = 256;
constexpr uint32_t kPanelMaxWb = 4096;  // widest binned row the panel path takes
// carry[Wb] + tile[sb][Wb] (u32); the symbol buffer (u16, + 32 bytes of
// alignment slack) starts 16-byte aligned, as a bulk copy's destination must;
// then the mbarrier
__host__ __device__ inline uint32_t panel_sym_offset(uint32_t Wb, uint32_t sb) { return (4 * Wb * (sb + 1) + 15) & ~15u; }
__host__ __device__ inline uint32_t panel_sym_bytes(uint32_t Wb, uint32_t sb) { return (2 * Wb * sb + 32 + 15) & ~15u; }
__host__ __device__ inline uint32_t panel_smem_bytes(uint32_t Wb, uint32_t sb) {
  return panel_sym_offset(Wb, sb) + panel_sym_bytes(Wb, sb) + 16;
}
// A panel's rows may be split over blocks of `rows` binned rows (a multiple of sb),
// when a small batch has too few panels: a block then starts from the column sums
// of all rows above its own, taken from the frame's symbols (a sparse frame's
// lists, or a thread per column over the symbol array).
// One CSPAD-like frame: 26 -> 7.4 us.
template <bool kSums>
__global__ void __launch_bounds__(kPanelThreads, 8) k_dec_panel(DevParams p, Scratch s, DecArgs a, uint32_t sb,
                                                                uint32_t rows, uint32_t lg_seg, int vec4) {
  chain_wait();
  extern __shared__ __align__(16) int32_t sm[];  // carry[Wb], tile[sb][Wb], symbols, mbarrier
  __shared__ int go;
  const uint32_t pn = blockIdx.x, f = blockIdx.y;
  const uint32_t Wb = p.Wb, Hb = p.Hb, Mp = Hb * Wb, W = p.W, H = p.H, bh = p.bh;
  if (threadIdx.x == 0) {
    go = s.status[f] == ROIBIN_OK && s.dec_zero[f] == s.dec_info[f].pl.n_lo;
    // a code-0 count that differs from the Lorenzo-outlier count
    if (!go && s.status[f] == ROIBIN_OK) mark_corrupt(s, f);
    // the bulk copy's destination must be 16-byte aligned
    if ((smem_u32(reinterpret_cast<uint8_t*>(sm) + panel_sym_offset(Wb, sb)) & 15u) != 0) {
      go = 0;
      s.status[f] = ROIBIN_ERR_CUDA;
    }
  }
  __syncthreads();
  if (!go) return;
  const DecInfo& di = s.dec_info[f];
  const uint32_t pb = pn * Mp;
  const int32_t R = di.R;
  const float two_eb = di.two_eb;
  const uint8_t* base = a.in + di.base;
  const uint2* lo = reinterpret_cast<const uint2*>(base + di.pl.off_lo);
  const uint2* pq = reinterpret_cast<const uint2*>(base + di.pl.off_pq);
  const uint32_t* lo_start = dec_list_starts(s, p, f);
  const uint32_t* pq_start = lo_start + p.P;
  uint32_t lo_cur = lo_start[pn], pq_cur = pq_start[pn];
  uint32_t lo_end = pn + 1 < p.P ? lo_start[pn + 1] : di.pl.n_lo;
  uint32_t pq_end = pn + 1 < p.P ? pq_start[pn + 1] : di.pl.n_pq;
  const uint32_t row0 = blockIdx.z * rows, row1 = min(Hb, row0 + rows);  // the block's binned rows
  const uint32_t lo_first = lo_cur;
  if (gridDim.z > 1) {  // the block's part of the panel's outliers
    auto below = [&](const uint2* v, uint32_t from, uint32_t to, uint32_t bin) {  // first entry at or past bin
      while (from < to) {
        const uint32_t mid = (from + to) >> 1;
        if (v[mid].x < bin) from = mid + 1;
        else to = mid;
      }
      return from;
    };
    const uint32_t b0 = pb + row0 * Wb, b1 = pb + row1 * Wb;
    lo_end = below(lo, lo_cur, lo_end, b1);
    lo_cur = below(lo, lo_cur, lo_end, b0);
    pq_end = below(pq, pq_cur, pq_end, b1);
    pq_cur = below(pq, pq_cur, pq_end, b0);
  }
  uint32_t* carry = reinterpret_cast<uint32_t*>(sm);
  uint32_t* tile = carry + Wb;
  float* tilef = reinterpret_cast<float*>(tile);
  uint8_t* symbuf = reinterpret_cast<uint8_t*>(sm) + panel_sym_offset(Wb, sb);
  uint64_t* bar = reinterpret_cast<uint64_t*>(symbuf + panel_sym_bytes(Wb, sb));
  // the frame's symbols start 16-byte aligned (chunks of kChunk u16)
  const uint8_t* fsym = reinterpret_cast<const uint8_t*>(s.codes + (size_t)f * p.n_chunks * kChunk);
  const uint64_t policy = evict_first_policy();
  // strip r0's symbols: bytes [2 (pb + r0 Wb), 2 (pb + (r0 + nr) Wb)) of fsym,
  // copied from the 16-byte boundary below to the one above
  auto fetch = [&](uint32_t r0) {
    const uint32_t nr = min(sb, row1 - r0);
    const uint32_t b0 = 2 * (pb + r0 * Wb), b1 = 2 * (pb + (r0 + nr) * Wb);
    const uint32_t a0 = b0 & ~15u, a1 = (b1 + 15) & ~15u;
    fence_proxy_async();
    mbar_expect_tx(bar, a1 - a0);
    tma_load_1d(symbuf, fsym + a0, a1 - a0, bar, policy);
  };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  // a sparse frame's strips are filled with the length-1 code's delta and its
  // listed symbols scattered in; a dense frame's symbols come by bulk copy
  const bool sparse = di.sparse != 0;
  const uint32_t zsym = s.dec_table[(size_t)f * kDecTableWords + 102];
  const uint32_t fillv = zsym ? (uint32_t)((int32_t)zsym - R) : (uint32_t)kSentinel;
  const uint32_t* counts = dec_list_count(s, p, f);
  if (threadIdx.x == 0 && !sparse) fetch(row0);
  uint32_t phase = 0;
  bool timed_out = false;  // uniform: set after a barrier
  float* panel = a.out + (size_t)f * p.frame_px + (size_t)pn * H * W;
  // row-segment role: row seg_row of the strip, segment seg of 2^lg_seg
  const uint32_t G = 1u << lg_seg, seg_row = threadIdx.x >> lg_seg, seg = threadIdx.x & (G - 1);
  const uint32_t seg_len = ceil_div(Wb, G);
  const uint32_t sj0 = min(Wb, seg * seg_len), sj1 = min(Wb, sj0 + seg_len);
  // output role (vec4): float4 column c4 of bin row orow, advanced by (dr, dc)
  const uint32_t W4 = W / 4;
  const uint32_t dr = vec4 ? blockDim.x / W4 : 0, dc = vec4 ? blockDim.x - dr * W4 : 0;
  bool bad = false;
  const uint32_t lane = lane_id();
  // column sums of the rows above the block's
  const uint32_t above = pb + row0 * Wb;  // bins pb .. above - 1
  if (sparse || row0 == 0) {
    for (uint32_t j = threadIdx.x; j < Wb; j += blockDim.x) carry[j] = fillv * row0;
    __syncthreads();
    if (row0 > 0) {
      // the listed symbols in place of the fill; a code 0's value is its outlier's
      for (uint32_t k = pb / kChunk; k <= (above - 1) / kChunk; ++k) {
        const uint32_t* list = dec_list(s, p, f, k);
        const uint32_t cnt = min(counts[k], kDecSparseMax), kb = k * kChunk;
        for (uint32_t e = threadIdx.x; e < cnt; e += blockDim.x) {
          const uint32_t v = list[e], x = kb + (v >> 16), u = v & 0xFFFFu;
          if (x >= pb && x < above)
            atomicAdd(carry + (x - pb) % Wb, (u ? (uint32_t)((int32_t)u - R) : (uint32_t)kSentinel) - fillv);
        }
      }
    }
  } else {
    const uint16_t* u16 = reinterpret_cast<const uint16_t*>(fsym) + pb;
    for (uint32_t j = threadIdx.x; j < Wb; j += blockDim.x) {
      uint32_t q = 0;
#pragma unroll 8
      for (uint32_t i = 0; i < row0; ++i) {
        const uint32_t u = __ldg(u16 + (size_t)i * Wb + j);
        q += u ? (uint32_t)((int32_t)u - R) : (uint32_t)kSentinel;
      }
      carry[j] = q;
    }
    __syncthreads();
  }
  if (row0 > 0)  // outliers above: the sentinel's value goes
    for (uint32_t e = lo_first + threadIdx.x; e < lo_cur; e += blockDim.x) {
      const uint2 x = lo[e];
      if (x.x >= pb) atomicAdd(carry + (x.x - pb) % Wb, x.y - (uint32_t)kSentinel);
      else bad = true;
    }
  __syncthreads();
  for (uint32_t r0 = row0; r0 < row1; r0 += sb) {
    const uint32_t nr = min(sb, row1 - r0), nb = nr * Wb;
    const uint32_t sb0 = pb + r0 * Wb, sb1 = sb0 + nb;
    // symbols -> deltas (code 0: sentinel until its outlier arrives)
    if (sparse) {
      for (uint32_t e = threadIdx.x; e < nb; e += blockDim.x) tile[e] = fillv;
      __syncthreads();
      // the strip's bins lie in chunks sb0 / kChunk .. (sb1 - 1) / kChunk
      for (uint32_t k = sb0 / kChunk; k <= (sb1 - 1) / kChunk; ++k) {
        const uint32_t* list = dec_list(s, p, f, k);
        const uint32_t cnt = min(counts[k], kDecSparseMax), kb = k * kChunk;
        for (uint32_t e = threadIdx.x; e < cnt; e += blockDim.x) {
          const uint32_t v = list[e], x = kb + (v >> 16), u = v & 0xFFFFu;
          if (x >= sb0 && x < sb1) tile[x - sb0] = u ? (uint32_t)((int32_t)u - R) : (uint32_t)kSentinel;
        }
      }
      __syncthreads();
    } else {
      const bool late = !mbar_wait(bar, phase);
      phase ^= 1u;
      if (!late) {
        const uint16_t* u16 = reinterpret_cast<const uint16_t*>(symbuf) + ((2 * (pb + r0 * Wb)) & 15u) / 2;
        for (uint32_t e = threadIdx.x; e < nb; e += blockDim.x) {
          const uint32_t u = u16[e];
          tile[e] = u ? (uint32_t)((int32_t)u - R) : (uint32_t)kSentinel;
        }
      }
      if (__syncthreads_or(late)) {
        // a copy that did not land in time: wait for it once more (bounded), then stop
        if (threadIdx.x == 0) mbar_wait(bar, phase ^ 1u);
        timed_out = true;
        break;
      }
      // the buffer is free: the next strip's symbols come in behind this one
      if (threadIdx.x == 0 && r0 + sb < row1) fetch(r0 + sb);
    }
    if (lo_cur != lo_end)
      lo_cur = place_strip_outliers(lo, lo_cur, lo_end, sb1, [&](uint32_t x, uint32_t y) {
      if (x < sb0 || tile[x - sb0] != (uint32_t)kSentinel) return false;
      tile[x - sb0] = y;
      return true;
    }, bad);
    // column prefix sums, carried from the strip above (unsigned: wraps instead
    // of overflowing on corrupt input)
    for (uint32_t j = threadIdx.x; j < Wb; j += blockDim.x) {
      uint32_t q = carry[j];
      for (uint32_t i = 0; i < nr; ++i) {
        q += tile[i * Wb + j];
        tile[i * Wb + j] = q;
      }
      carry[j] = q;
    }
    __syncthreads();
    // prequantisation outliers in this strip (the same answer in every thread)
    const bool any_pq = !kSums && pq_cur != pq_end && pq[pq_cur].x < sb1;
    if constexpr (kSums) {
      // a warp per row, two bins a lane, as below
      uint32_t* out = reinterpret_cast<uint32_t*>(s.dq) + (size_t)f * p.M + sb0;
      for (uint32_t i = threadIdx.x >> 5; i < nr; i += kPanelThreads / 32) {
        const uint32_t* row = tile + i * Wb;
        uint32_t run = 0;
        for (uint32_t j0 = 0; j0 < Wb; j0 += 64) {
          const uint32_t j = j0 + 2 * lane;
          const uint32_t x = j < Wb ? row[j] : 0u, y = j + 1 < Wb ? row[j + 1] : 0u;
          const uint32_t incl = warp_incl_scan(x + y);
          const uint32_t q0 = run + incl - y, q1 = run + incl;
          run += __shfl_sync(0xffffffffu, incl, 31);
          if (vec4) {  // even rows and panels: 8-byte aligned
            if (j < Wb) *reinterpret_cast<uint2*>(out + i * Wb + j) = make_uint2(q0, q1);
          } else {
            if (j < Wb) out[i * Wb + j] = q0;
            if (j + 1 < Wb) out[i * Wb + j + 1] = q1;
          }
        }
      }
    } else if (vec4 && !any_pq) {
      // a warp per row: row prefix sums by shuffles, two bins a lane, and from the
      // registers b^ = fl(q * 2eb) straight to the row's pixels (one float4 on each
      // of its pixel rows; streaming stores: the kernel never reads them back)
      for (uint32_t i = threadIdx.x >> 5; i < nr; i += kPanelThreads / 32) {
        const uint2* row = reinterpret_cast<const uint2*>(tile + i * Wb);
        const uint32_t pr0 = (r0 + i) * bh, pr1 = min(H, pr0 + bh);
        float4* px = reinterpret_cast<float4*>(panel + (size_t)pr0 * W);
        uint32_t run = 0;  // sum of the row before this round's bins
        for (uint32_t c0 = 0; c0 < W4; c0 += 32) {
          const uint32_t c4 = c0 + lane;
          const uint2 v = c4 < W4 ? row[c4] : make_uint2(0u, 0u);
          const uint32_t sum = v.x + v.y, incl = warp_incl_scan(sum);
          const uint32_t q0 = run + incl - v.y, q1 = run + incl;
          run += __shfl_sync(0xffffffffu, incl, 31);
          if (c4 < W4) {
            const float b0 = __fmul_rn((float)(int32_t)q0, two_eb), b1 = __fmul_rn((float)(int32_t)q1, two_eb);
            const float4 o = make_float4(b0, b0, b1, b1);
            for (uint32_t pr = pr0; pr < pr1; ++pr) __stcs(px + (size_t)(pr - pr0) * W4 + c4, o);
          }
        }
      }
    } else {
      // row prefix sums and b^ = fl(q * 2eb)
      {
        const bool mine = seg_row < nr;
        uint32_t* row = tile + seg_row * Wb;
        uint32_t run = 0;
        if (mine)
          for (uint32_t j = sj0; j < sj1; ++j) {
            run += row[j];
            row[j] = run;
          }
        // exclusive scan of the segment totals across the G lanes of the row
        uint32_t incl = run;
        for (uint32_t d = 1; d < G; d <<= 1) {
          const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d, G);
          if (seg >= d) incl += v;
        }
        const uint32_t excl = incl - run;
        if (mine)
          for (uint32_t j = sj0; j < sj1; ++j)
            tilef[seg_row * Wb + j] = __fmul_rn((float)(int32_t)(row[j] + excl), two_eb);
      }
      __syncthreads();
      pq_cur = place_strip_outliers(pq, pq_cur, pq_end, sb1, [&](uint32_t x, uint32_t y) {
        if (x < sb0) return false;
        tilef[x - sb0] = __uint_as_float(y);
        return true;
      }, bad);
      // output rows of the strip: bin row i covers pixel rows (r0 + i) * bh ...
      // (streaming stores: the kernel never reads these pixels back)
      if (vec4) {  // bin width 2, W % 4 == 0: one float4 = 2 bins, stored on each of its rows
        const uint32_t n2 = nr * W4;
        uint32_t i = threadIdx.x / W4, c4 = threadIdx.x - i * W4;
        for (uint32_t e = threadIdx.x; e < n2; e += blockDim.x) {
          const float2 v = *reinterpret_cast<const float2*>(tilef + i * Wb + 2 * c4);
          const float4 o = make_float4(v.x, v.x, v.y, v.y);
          const uint32_t pr0 = (r0 + i) * bh, pr1 = min(H, pr0 + bh);
          for (uint32_t pr = pr0; pr < pr1; ++pr) __stcs(reinterpret_cast<float4*>(panel + (size_t)pr * W) + c4, o);
          i += dr;
          c4 += dc;
          if (c4 >= W4) {
            c4 -= W4;
            ++i;
          }
        }
      } else {
        const uint32_t ro0 = r0 * bh, ro1 = min(H, (r0 + nr) * bh);
        const uint32_t n1 = (ro1 - ro0) * W;
        for (uint32_t e = threadIdx.x; e < n1; e += blockDim.x) {
          const uint32_t rr = e / W, c = e - rr * W;
          __stcs(panel + (size_t)ro0 * W + e, tilef[((ro0 + rr) / bh - r0) * Wb + c / p.bw]);
        }
      }
    }
    __syncthreads();
  }
  if (lo_cur != lo_end || (!kSums && pq_cur != pq_end)) bad = true;
  if (timed_out) {
    if (threadIdx.x == 0) s.status[f] = ROIBIN_ERR_TIMEOUT;
    return;
  }
  if (bad) mark_corrupt(s, f);
}

// ROI mask: u8 per pixel, 1 on every in-panel pixel of some peak's window.
__global__ void k_roi_mask_set(DevParams p, const uint16_t* peaks, const uint32_t* npeaks, uint8_t* mask) {
  const uint32_t f = blockIdx.y;
  const uint32_t n = min(npeaks[f], p.max_peaks);
  const uint32_t k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k >= n) return;
  const uint16_t* pk = peaks + ((size_t)f * p.max_peaks + k) * 3;
  const uint32_t pn = pk[0], r = pk[1], c = pk[2];
  if (pn >= p.P || r >= p.H || c >= p.W) return;
  uint8_t* m = mask + (size_t)f * p.frame_px + (size_t)pn * p.H * p.W;
  const int r0 = (int)r - p.roi_h / 2, c0 = (int)c - p.roi_w / 2;
  const uint32_t win = (uint32_t)(p.roi_h * p.roi_w);
  for (uint32_t e = lane_id(); e < win; e += 32) {
    const int rr = r0 + (int)(e / p.roi_w), cc = c0 + (int)(e % p.roi_w);
    if (rr >= 0 && rr < (int)p.H && cc >= 0 && cc < (int)p.W) m[(size_t)rr * p.W + cc] = 1;
  }
}

// pack: copy each frame's stream from its strided slot to its packed offset.
__global__ void k_pack(const uint8_t* src, uint64_t stride, const uint64_t* sizes,
                       const uint64_t* offsets, uint8_t* dst) {
  const uint32_t f = blockIdx.y;
  const uint64_t n16 = sizes[f] / 16;
  const uint4* s4 = reinterpret_cast<const uint4*>(src + (size_t)f * stride);
  uint4* d4 = reinterpret_cast<uint4*>(dst + offsets[f]);
  for (uint64_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n16; e += (uint64_t)gridDim.x * blockDim.x)
    d4[e] = s4[e];
}

// ---------------------------------------------------------------------------
cudaError_t launch_dec_parse(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  return launch_chained(k_dec_parse, a.n_frames, 256, 0, st, p, s, a);
}
cudaError_t launch_dec_decode(const DevParams& p, const Scratch& s, const DecArgs& a, bool deltas, cudaStream_t st) {
  // dense blocks: one round of chunks each while that is at most two waves of 304
  // resident blocks, else as many rounds as bring it there (each block builds its
  // tables once, and the blocks of sparse frames end at once)
  const uint32_t rounds = std::max<uint32_t>(1, (uint32_t)((uint64_t)ceil_div(p.n_chunks, kDecWarps) * a.n_frames / 608));
  const dim3 grid(ceil_div(ceil_div(p.n_chunks, kDecWarps), rounds), a.n_frames);
  const auto dense = deltas ? k_dec_dense<true> : k_dec_dense<false>;
  cudaError_t e = allow_smem(dense, 1024);
  if (e != cudaSuccess) return e;
  if (deltas) return launch_chained(dense, grid, kDecWarps * 32, kDecSmem, st, p, s, a);
  // sparse blocks: as many chunks per warp as bring them to 2,432 (six are resident per
  // SM, 912 in all), since each block loads the frame's tables (13 KB).  CSPAD-like frames, caches
  // flushed, 1 / 2 / 3 / 9 chunks per warp: 16 frames 16 / 22 / 25 / 48 us, 200 frames
  // 39 / 35 / 39 / 64 us, 400 frames 67 / 58 / 57 / 67 us, 1,000 frames 165 / 134 / 126 / 124 us
  const uint32_t blocks = ceil_div(p.n_chunks, kDecWarps);
  const uint32_t per = std::max<uint32_t>(1, (uint32_t)(((uint64_t)blocks * a.n_frames + 2431) / 2432));
  e = launch_chained(k_dec_sparse, dim3(ceil_div(blocks, per), a.n_frames), kDecWarps * 32, 0, st, p, s, a);
  if (e != cudaSuccess) return e;
  return launch_chained(dense, grid, kDecWarps * 32, kDecSmem, st, p, s, a);
}
cudaError_t launch_dec_lorenzo(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  dim3 grid(64, a.n_frames);
  return launch_chained(k_dec_lorenzo, grid, 256, 0, st, p, s, a);
}
cudaError_t launch_dec_rows(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  dim3 grid(ceil_div(p.P * p.Hb, 8), a.n_frames);
  return launch_chained(k_dec_rows, grid, 256, 0, st, p, s, a);
}
cudaError_t launch_dec_cols(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  dim3 grid(ceil_div(p.P * p.Wb, 128), a.n_frames);
  return launch_chained(k_dec_cols, grid, 128, 0, st, p, s, a, p.dims == 2 ? 1 : 0);
}
cudaError_t launch_dec_carry(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  return launch_chained(k_dec_chain, a.n_frames, kChainThreads, 0, st, p, s, a);
}
cudaError_t launch_dec_stack_out(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  const bool vec = p.bh == 2 && p.bw == 2 && (p.W % 4) == 0 && (reinterpret_cast<uintptr_t>(a.out) % 16) == 0;
  const dim3 grid(ceil_div(p.Hb * (vec ? p.W / 4 : p.W), 256), a.n_frames);
  return launch_chained(vec ? k_dec_stack_out<true> : k_dec_stack_out<false>, grid, 256, 0, st, p, s, a);
}
cudaError_t launch_dec_pq_pixels(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  return launch_chained(k_dec_pq_pixels, dim3(16, a.n_frames), 256, 0, st, p, s, a);
}
cudaError_t launch_dec_pq(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  dim3 grid(16, a.n_frames);
  return launch_chained(k_dec_pq, grid, 256, 0, st, p, s, a);
}
cudaError_t launch_dec_upsample(const DevParams& p, const Scratch& s, const DecArgs& a, cudaStream_t st) {
  const bool vec4 = p.bh == 2 && p.bw == 2 && (p.W % 4) == 0 && (p.Wb % 2) == 0 &&
                    (reinterpret_cast<uintptr_t>(a.out) % 16) == 0;
  dim3 grid(ceil_div((uint32_t)(p.frame_px / 4 / 256), 4) + 1, a.n_frames);
  return launch_chained(k_dec_upsample, grid, 256, 0, st, p, s, a, vec4 ? 1 : 0);
}
uint32_t dec_panel_rows(const DevParams& p) {
  if (p.Wb > kPanelMaxWb) return 0;
  // the most rows (up to 32) that fit 24 KB, so that 8 blocks share an SM
  // (at least one row, in up to 48 KB), then evened out over the strips
  uint32_t most = 1;
  while (most < 32 && most < p.Hb && panel_smem_bytes(p.Wb, most + 1) <= 24576) ++most;
  const uint32_t strips = ceil_div(p.Hb, most);
  return ceil_div(p.Hb, strips);
}
cudaError_t launch_dec_panel(const DevParams& p, const Scratch& s, const DecArgs& a, bool sums, cudaStream_t st) {
  uint32_t sb = dec_panel_rows(p);
  if (sb == 0) return cudaErrorInvalidValue;
  // few panels: strips of fewer rows, a block each, until about four blocks an SM
  // have work (at least four rows, as every block reads the symbols above its own)
  uint32_t rows = p.Hb;
  const uint32_t panels = p.P * a.n_frames;
  if (panels < 304) {
    const uint32_t parts = std::max<uint32_t>(1, std::min<uint32_t>(608 / panels, p.Hb / 4));
    rows = ceil_div(p.Hb, parts);
    sb = ceil_div(rows, ceil_div(rows, sb));
    rows = ceil_div(rows, sb) * sb;
  }
  // sums: pairs of them are stored together when the binned rows are even
  const bool vec4 = sums ? (p.Wb % 2) == 0 : p.bw == 2 && (p.W % 4) == 0 && (reinterpret_cast<uintptr_t>(a.out) % 16) == 0;
  const size_t smem = panel_smem_bytes(p.Wb, sb);
  // row segments: the most lanes per row that still give every row of a strip
  // its own lanes (sb <= 32, so at least 8)
  uint32_t lg_seg = 5;
  while (lg_seg > 0 && (sb << lg_seg) > (uint32_t)kPanelThreads) --lg_seg;
  dim3 grid(p.P, a.n_frames, ceil_div(p.Hb, rows));
  return launch_chained(sums ? k_dec_panel<true> : k_dec_panel<false>, grid, kPanelThreads, smem, st, p, s, a, sb, rows,
                        lg_seg, vec4 ? 1 : 0);
}
cudaError_t launch_roi_mask(const DevParams& p, const uint16_t* peaks, const uint32_t* npeaks, uint32_t n,
                            uint8_t* mask, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(mask, 0, (size_t)n * p.frame_px, st);
  if (e != cudaSuccess || p.max_peaks == 0) return e;
  dim3 grid(ceil_div(p.max_peaks, 8), n);
  k_roi_mask_set<<<grid, 256, 0, st>>>(p, peaks, npeaks, mask);
  return cudaGetLastError();
}
cudaError_t launch_pack(const uint8_t* src, uint64_t stride, const uint64_t* sizes, const uint64_t* offsets,
                        uint32_t n, uint8_t* dst, cudaStream_t st) {
  dim3 grid(64, n);
  k_pack<<<grid, 256, 0, st>>>(src, stride, sizes, offsets, dst);
  return cudaGetLastError();
}

}  // namespace roibin
