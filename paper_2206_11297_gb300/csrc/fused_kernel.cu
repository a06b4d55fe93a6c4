// fused_kernel.cu - the persistent batched kernel: the whole method for a
// batch of frames in one launch.
//
// Work items are handed out in order by an atomic ticket counter to a grid of
// resident CTAs (several per SM).  A streaming item is a group of k panels of
// one frame side by side (k NP <= 217 kG float4 columns, NP = cols / 4, kG
// column groups of 217: 1, or 2 for panels wider than 868 columns).  For it
// a CTA:
//   - streams the raw rows through a ring of 1-D TMA bulk copies (L2
//     evict-first) while the previous rows are coded;
//   - walks down the rows with one thread per float4 column (two bins per
//     binned row): bins, prequantises, predicts with the 2-D Lorenzo rule from
//     registers (row above) and shuffles (bin to the left) and writes one byte
//     per bin (byte = residual + 128 for residuals in [-127, 126], 0 = Lorenzo
//     outlier, 255 = escape whose code sits in a side array);
//   - keeps the item's histogram, prequantisation outliers and the 2x4 blocks
//     holding a pixel >= amax_thr in shared memory, adds the histogram to the
//     frame's and writes the outliers' bits to a slot per panel and band;
//   - prunes the listed blocks' candidates, tests and evaluates the others and adds
//     its peaks to the frame's list (the codebook stage sorts it).
// In small batches an item is a band of rows of its panels (band_shape).
// The rest of a frame's work (codebook, chunk sizes, layout, bit-packing)
// runs as later work items of the same kernel (see the stages below), after the
// whole batch has streamed; a codebook is built by the CTA that completes its frame.
// After use, a frame's code bytes are dropped from L2 without a write-back.
#include <algorithm>

#include "fused_device.cuh"

namespace roibin {

// ---------------------------------------------------------------------------
// host side
__global__ void k_sync_reset(uint32_t* words, uint32_t n) {
  chain_wait();
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) words[i] = 0;
}

// The candidates of an item up to which they are tested a warp each (eight at a time,
// about 5 us a round); above, they are tested a lane each, band by band (a few us a band
// of rows in shared memory).  100 CSPAD-like frames (32 bands an item) with 0.2, 0.3 and
// 0.4% of hot pixels, 7 / 10 / 14 / 20 candidates a band: 1,253 / 1,646 / 1,640 / 1,646 us,
// 1,380 / 1,375 / 2,216 / 2,216 us, 1,385 / 1,477 / 1,487 / 2,712 us; with 0.15%, 7 cost
// 1,434 us and the others 1,350 us.
static void set_list_max(const DevParams& p, FusedShape* sh) {
  if (!sh->band_rows) {
    sh->list_max = kThrLocalCap + kThrSpill;
    return;
  }
  const uint32_t own = sh->band_rows - 2 * (uint32_t)peak_reach(p);  // rows a band adds
  const uint32_t bands = sh->k * ceil_div(min(p.H, 2 * sh->band_bins), own);
  sh->list_max = min(10u * bands, kThrLocalCap + kThrSpill);
}

// Shared memory a CTA of this shape needs (0 if the shape is impossible).
static bool make_shape(const DevParams& p, uint32_t ctas_per_sm, uint32_t rb, uint32_t stages, FusedShape* out) {
  FusedShape sh{};
  const uint32_t NP = p.W / 4;
  if (NP < 1 || NP > kMaxG * kGroupCols || rb < 2 || rb > 3) return false;
  sh.kG = ceil_div(NP, kGroupCols);
  if (sh.kG > 1 && rb != 2) return false;  // wide panels: two binned rows per step
  sh.k = min(kMaxK, sh.kG * kGroupCols / NP);
  if ((uint64_t)sh.k * p.H * p.W >= kBlockKey) return false;  // item-local keys stay below the flag
  sh.U = ceil_div(p.P, sh.k);
  sh.stack = p.dims == 3 ? ceil_div(p.Hb * p.Wb, kStackSlice) : 0u;
  sh.bands = 1;
  sh.band_bins = p.Hb;
  sh.RB = rb;
  sh.stages = stages;
  // the streamed rows are read once: first out of L2, so that the code bytes
  // (evict-last) stay there longer (1,000 CSPAD-like frames: +1%)
  sh.input_evict_first = 1;
  sh.wait_limit = kWaitLimit;
  sh.stage_bytes = sh.k * 2 * rb * p.W * 4;
  sh.ctas_per_sm = ctas_per_sm;
  sh.mask_words = ceil_div(p.Hb * p.Wb, 32) + 1;
  sh.side = 2 * (uint32_t)peak_reach(p) + 1;
  uint32_t n2 = 4;  // words the peak sort needs
  while (n2 < p.max_peaks) n2 <<= 1;
  sh.n_chunks = p.n_chunks;
  sh.codes_stride = p.n_chunks * kChunk;
  sh.group_chunks = 2 * kPW;
  sh.groups = ceil_div(p.n_chunks, sh.group_chunks);
  uint64_t off = 0;
  auto take = [&](uint64_t bytes) {
    off = (off + 15) / 16 * 16;
    const uint64_t o = off;
    off += bytes;
    return (uint32_t)o;
  };
  sh.off_ctl = take((uint64_t)CTL_WORDS * 4);  // every role uses the control words
  sh.off_bar = take(16ull * stages + 8);  // ring full / empty barriers, then the band barrier
  const uint64_t base = off;
  // streaming role; the peak tests reuse the ring once the rows are consumed
  sh.off_hist = take(kMaxSymbols * 4);
  sh.off_pql = take(kPqList * 4);
  sh.off_thr = take(kThrLocalCap * 8);  // keys, then values
  off = (off + 127) / 128 * 128;
  sh.off_ring = take((uint64_t)stages * sh.stage_bytes);
  const uint64_t ring_end = off;
  off = sh.off_ring;
  sh.off_nb = take((uint64_t)kPW * sh.side * sh.side * 4);
  sh.off_cand = take(kThrLocalCap * 4);
  const uint64_t stream_end = off > ring_end ? off : ring_end;
  // codebook role / size, write and plan roles (overlap the streaming role)
  off = base;
  sh.off_huff = take(kHuffArea);  // Huffman scratch | byte tables | slices of the 3-D stacking
  const uint64_t after_huff = off;
  off = sh.off_huff + 4096;  // chunk staging of the size and write items (after the byte tables)
  sh.off_stage = take((uint64_t)kPW * kStageWords * 4);
  const uint64_t stage_end = off;
  off = after_huff;
  sh.off_total = take(kMaxSymbols * 4);
  sh.off_cblen = take(kMaxSymbols);
  sh.off_cbcode = take(kMaxSymbols * 4);
  sh.off_cw = take(3ull * p.n_chunks * 4);
  const uint64_t sort_end = sh.off_huff + (uint64_t)n2 * 4;  // before the histogram is read
  uint64_t fin_end = off > stage_end ? off : stage_end;
  if (sort_end > fin_end) fin_end = sort_end;
  sh.smem = (uint32_t)(stream_end > fin_end ? stream_end : fin_end);
  // The dense-peaks variant takes all the shared memory its CTAs per SM leave
  // it: from the ring on, that memory holds a band of rows of one panel once
  // the item's rows are coded.  A band's candidates are tested in parallel, one
  // per thread, so a taller band keeps more threads busy.
  const uint32_t share = 233472u / ctas_per_sm - 1024u;
  // A large neighbourhood leaves such a band few rows of its own: it also takes what the
  // warp tests' buffers and a frame's list of peaks need, at the cost of a CTA (31 x 31 and
  // 8,192 peaks at 388 columns: 11 rows instead of 2; 100 frames with 1% of hot pixels
  // 45.6 -> 13.0 ms).
  const uint64_t tests = sh.off_ring + (uint64_t)kPW * sh.side * sh.side * 4 + (uint64_t)n2 * 4 + kThrLocalCap * 4;
  const uint32_t room = (uint32_t)std::min<uint64_t>(kBlockSmem, std::max<uint64_t>(share, tests));
  sh.smem_dense = sh.smem > room ? sh.smem : room;
  const uint32_t least = 2 * (uint32_t)peak_reach(p) + 2;
  auto rows_in = [&](uint32_t smem) {
    const uint32_t rows = (smem - sh.off_ring) / (p.W * 4);
    return rows >= least ? rows : 0u;
  };
  sh.band_rows = rows_in(sh.smem);
  sh.band_rows_dense = rows_in(sh.smem_dense);
  set_list_max(p, &sh);
  *out = sh;
  return sh.smem <= kBlockSmem;
}

// The kernel instantiation for a shape: column groups, rows per step, row bands.
static FusedKernel fused_kernel(const FusedShape& sh) {
  if (sh.bands > 1) return fused_band_kernel(sh.kG);
  if (sh.kG > 1) return k_fused<kMaxG, 2, false>;
  return sh.RB == 3 ? k_fused<1, 3, false> : k_fused<1, 2, false>;
}

bool fused_shape_for(const DevParams& p, uint32_t ctas_per_sm, uint32_t rows_per_step, uint32_t stages,
                     FusedShape* out) {
  // the 2-D predictor, or the 3-D one (the 2-D residuals stacked by items of their own)
  if (p.dims < 2 || p.bh != 2 || p.bw != 2 || (p.W % 4) != 0 || p.W / 4 > kMaxG * kGroupCols) return false;
  if (ctas_per_sm < 1 || ctas_per_sm > 8 || stages < 1 || stages > 8) return false;
  if (rows_per_step != 0 && (rows_per_step < 2 || rows_per_step > 3)) return false;
  FusedShape sh;
  bool ok = false;
  if (rows_per_step) {
    ok = make_shape(p, ctas_per_sm, rows_per_step, stages, &sh);
  } else {
    // the most rows per step whose shared memory lets ctas_per_sm CTAs share an SM
    const uint32_t budget = 233472u / ctas_per_sm - 1024u;
    for (uint32_t rb = 3; rb >= 2 && !ok; --rb) ok = make_shape(p, ctas_per_sm, rb, stages, &sh) && sh.smem <= budget;
  }
  if (!ok) return false;
  const FusedKernel kern = fused_kernel(sh);
  if (allow_smem(kern) != cudaSuccess) return false;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPT, sh.smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return false;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  sh.ctas_per_sm = min((uint32_t)per_sm, ctas_per_sm);
  sh.n_ctas = sh.ctas_per_sm * (uint32_t)sms;
  *out = sh;
  return true;
}

bool fused_plan(const DevParams& p, int device, int num_sms, FusedShape* out) {
  (void)device;
  (void)num_sms;
  // measured on CSPAD-like frames: 2 binned rows per step through a 3-slot
  // ring, 4 CTAs per SM, is the fastest shape that fits
  return fused_shape_for(p, 4, 2, 3, out) || fused_shape_for(p, 4, 2, 2, out) || fused_shape_for(p, 3, 2, 3, out) ||
         fused_shape_for(p, 2, 2, 2, out) || fused_shape_for(p, 1, 2, 1, out);
}

// Cuts the panels of a small batch into row bands: a batch of few frames has too
// few panel groups to occupy every CTA (one CSPAD frame has 16 for 608), and the
// last wave of a middling one is long.  The bands per panel with the least
//   waves x (an item's pixels per raw row pair x its binned rows + a fixed cost)
// where the fixed cost of an item (its start, flush and peak tests, about 12 us)
// is worth 17,000 of those pixels (a 776-pixel binned row takes 0.54 us), waves =
// items / CTAs (at least 1), and a partly filled wave after the first costs 0.15
// more.  us per call, whole panels -> bands: 1 CSPAD frame 93 -> 61, 8 frames 105
// -> 79, 16 frames 121 -> 96, 33 frames one band (132; two 147); 8 x 512 x 1024
// panels: 1 frame 291 -> 72, 5 frames 308 -> 100, 20 frames 430 -> 199, 60 frames
// 474 -> 430; 30 hot-pixel frames 1,120 -> 800, 100 of them one band (1,636; two
// 1,772).
static void band_shape(const DevParams& p, const Scratch& s, uint32_t n, FusedShape* sh) {
  const uint64_t items = (uint64_t)n * sh->U;
  if (sh->RB != 2 || items >= 4ull * sh->n_ctas) return;
  uint32_t best = p.Hb;
  double best_cost = 0.0;
  for (uint32_t bands = 1;; ++bands) {
    const uint32_t bins = (ceil_div(p.Hb, bands) + 1) & ~1u;  // whole steps of two rows
    if (bands > 1 && bins < 4) break;
    const double w = (double)items * ceil_div(p.Hb, bins) / sh->n_ctas;
    const double cost = (w > 1.0 ? w + 0.15 : 1.0) * ((double)min(bins, p.Hb) * sh->k * p.W + 17000.0);
    if (bands == 1 || cost < best_cost) {
      best = bins;
      best_cost = cost;
    }
    if (w > 4.0) break;  // more bands only add fixed costs
  }
  for (; best < p.Hb; best *= 2) {
    const uint32_t bands = ceil_div(p.Hb, best), words = ceil_div(best * p.Wb, 32) + 1;
    if ((uint64_t)n * p.P * bands * words > s.pq_mask_words) continue;  // the outlier slots do not fit
    sh->bands = bands;
    sh->band_bins = best;
    sh->mask_words = words;
    sh->U *= bands;
    set_list_max(p, sh);
    return;
  }
}

cudaError_t launch_fused(const DevParams& p, const Scratch& s, const PlainArgs& a, const FusedShape& sh,
                         bool dense, cudaStream_t st) {
  // stage counters, flags and the ticket counter start at zero (by a kernel, so that
  // the persistent one is set up meanwhile: a memset would end first)
  const uint32_t words = kSyncWordsPerFrame * a.n_frames + 1;
  cudaError_t e = launch_chained(k_sync_reset, min(ceil_div(words, 256), 32u), 256, 0, st, s.frame_done, words);
  if (e != cudaSuccess) return e;
  FusedShape s2 = sh;
  band_shape(p, s, a.n_frames, &s2);
  const uint32_t smem = dense ? sh.smem_dense : sh.smem;
  s2.dense = dense ? 1u : 0u;
  const FusedKernel kern = fused_kernel(s2);
  e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  // Every frame streams before any is sized: streaming is bound by the bytes each
  // CTA keeps in flight, and a CTA on a coding item has none (interleaving the
  // stages, 256 frames apart, ran 6% slower at 1,000 frames).  Chunk sizes ->
  // writing: 64 frames, so that a frame's plan is ready when its write items
  // come up.
  s2.lag = a.n_frames < kLagWrite ? a.n_frames : kLagWrite;
  const uint64_t tickets = fused_tickets(s2, a.n_frames);
  if (tickets + sh.n_ctas >= (1ull << 32)) return cudaErrorInvalidValue;
  const uint32_t grid = (uint32_t)(tickets < sh.n_ctas ? tickets : sh.n_ctas);
  return launch_chained(kern, grid, kPT, smem, st, p, s, a, s2);
}

}  // namespace roibin
