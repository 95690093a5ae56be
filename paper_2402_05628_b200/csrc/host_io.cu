// Host-buffer form of the block: a sequence of independent batches whose inputs and outputs live in host
// memory.  The copies and the block's kernels overlap through two device staging buffers per direction and two helper
// streams.  (Plumbing around the block; the block itself is repq_block_forward.)
//
// What bounds it is the host link: 53 GB/s in one direction, 44 GB/s in each when both are busy.  With whole batches the outputs
// run one batch behind the inputs, which costs a batch's time on the link and the block's own time at the end.  The items of a
// batch are independent, so a batch passes through the pipeline in pieces of whole items: piece c is computed while piece
// c + 1 is copied in and piece c - 1 copied out, and the outputs run one piece behind.  See `pieces_of` for when.
//
// Copies of the two directions begin together: the copy out of a piece waits for the next piece's copy in, and so starts with the one
// after it.  Where a copy begins while the other direction is under way the link stands for 10 us and more; with blocks shorter than
// their copies every copy did that to the other direction (six pieces of 3.2 MB: 100 us a piece, 76 while the two ran in step), and
// a faster block made a call slower.  Four batches of 64 DeiT-B images 2160 -> 1936 us, 20 of 40 ViT-S images, whole, 3790 -> 2860,
// four of 65 ViT-S images in float32 2590 -> 2030; 28 x 371 DeiT-B tokens and batches of 4.8 MB as before.  A single batch has too
// few copies to gain by it (64 DeiT-B images 580 us, 591 so): its pieces leave as their blocks end.
#include <algorithm>
#include <mutex>

#include "kernels.h"

namespace repq {
namespace {

constexpr int kMaxDevices = 64;
constexpr int kSlots = 2;
constexpr int kMaxPieces = 8;
constexpr size_t kPieceBytes = size_t(2685) << 10;       // 2.75 MB: 60 us of the link, a little more than queueing a piece takes the host
constexpr int64_t kPieceTokens = 2048;                   // (2765 with packed weights, whose expansion every piece repeats)
constexpr size_t kGapBytes = size_t(585) << 10;          // what the link would move while a further piece holds it up (14 us; copies
                                                         // alone stand 10 us apart, with the waits on events 10 to 25)

// Pieces per batch: as many as have kPieceBytes of input and kPieceTokens tokens each (below, the host, or the blocks of the pieces
// together, take longer than the link), unless what they save (the link time of a batch: the outputs no longer run a batch behind)
// is less than the gaps they add (one per piece and batch).
// Measured with every piece leaving as its block ended, us, whole -> pieces (ranges: different machines).  64 DeiT-B images of 19.4 MB, six pieces: one batch 935 -> 580, two
// 1340 -> 1092..1106, four 2240 -> 2083, five 2690 -> 2614..2638, eight 4051 -> 4194 (whole by the rule); four pieces: four 2250, five
// 2518..2833.  32 ViT-L images of 577 tokens, 37.8 MB, eight: 1841 -> 1029, four 4237 -> 3530, five 5065 -> 4362, sixteen 14157 -> 13644
// (whole).  16 of them, 18.9 MB, four: 955 -> 612, five 2655 -> 2280 (seven pieces, 1300 tokens each: 2894).  28 x 371 tokens of
// DeiT-B, 16 MB, five: two 1143 -> 922, five 2266 -> 2086.  64 x 133 with packed weights, 13.1 MB, three: 667 -> 467, five 1905 -> 1655
// (four pieces 1846).  100 x 50, 7.7 MB, two: 412 -> 316, five 1214 -> 1064.  4 x 2048 LLaMA tokens, 67 MB, four: five 9036..9373 ->
// 7841..7950, twenty 30340..32116 -> 31095..32195.  Batches of 4.8 MB stay whole: in two pieces four take 633 for 605.
// Pieces for the first and the last batch only gain nothing beyond two batches: the outputs then fall a batch behind in between.
int pieces_of(size_t x_bytes, const repq_block_desc& d, int n_batches) {
  const bool packed = packed4(d.bits_w) || packed6(d.bits_w);
  int64_t pieces = kMaxPieces;
  pieces = std::min(pieces, int64_t(x_bytes / kPieceBytes));
  pieces = std::min(pieces, int64_t(d.batch) * d.seq / (packed ? kPieceTokens * 27 / 20 : kPieceTokens));
  pieces = std::min(pieces, int64_t(d.batch));
  if (pieces < 2) return 1;
  return size_t(n_batches) * size_t(pieces) * kGapBytes <= x_bytes ? int(pieces) : 1;
}

struct Pipeline {                 // per device, created on first use, kept for the life of the process
  std::mutex queueing;            // held while a call queues its work: a wait on an event means its last record, and calls of
                                  // several threads record the same events
  bool ready = false;
  cudaStream_t in = nullptr, out = nullptr;
  cudaEvent_t start = nullptr;
  cudaEvent_t copied_in[kSlots][kMaxPieces] = {}, computed[kSlots][kMaxPieces] = {}, copied_out[kSlots][kMaxPieces] = {};
};
Pipeline g_pipe[kMaxDevices];
std::mutex g_pipe_mutex;

repq_status pipeline(Pipeline** out) {
  int dev = -1;
  REPQ_CUDA(cudaGetDevice(&dev));
  REPQ_REQUIRE(dev >= 0 && dev < kMaxDevices, REPQ_UNSUPPORTED, "block_forward_host: device index %d not supported", dev);
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  Pipeline& P = g_pipe[dev];
  if (!P.ready) {
    REPQ_CUDA(cudaStreamCreateWithFlags(&P.in, cudaStreamNonBlocking));
    REPQ_CUDA(cudaStreamCreateWithFlags(&P.out, cudaStreamNonBlocking));
    REPQ_CUDA(cudaEventCreateWithFlags(&P.start, cudaEventDisableTiming));
    for (int s = 0; s < kSlots; ++s)
      for (int c = 0; c < kMaxPieces; ++c) {
        REPQ_CUDA(cudaEventCreateWithFlags(&P.copied_in[s][c], cudaEventDisableTiming));
        REPQ_CUDA(cudaEventCreateWithFlags(&P.computed[s][c], cudaEventDisableTiming));
        REPQ_CUDA(cudaEventCreateWithFlags(&P.copied_out[s][c], cudaEventDisableTiming));
      }
    P.ready = true;
  }
  *out = &P;
  return REPQ_OK;
}

size_t dtype_size(int dtype) { return dtype == REPQ_F32 ? 4 : 2; }

}  // namespace
}  // namespace repq

using namespace repq;

extern "C" repq_status repq_block_forward_host(const repq_block_desc* d, const repq_block_params* p,
                                               const void* const* x_host, void* const* y_host, int n_batches,
                                               const repq_host_staging* s, void* stream) {
  REPQ_REQUIRE(d && p && x_host && y_host && s, REPQ_INVALID_ARG, "block_forward_host: NULL argument");
  REPQ_REQUIRE(n_batches >= 0, REPQ_INVALID_ARG, "block_forward_host: negative number of batches");
  REPQ_REQUIRE(d->act_dtype == REPQ_F32 || d->act_dtype == REPQ_BF16, REPQ_INVALID_ARG, "block_forward_host: bad act_dtype");
  REPQ_REQUIRE(d->out_dtype == REPQ_F32 || d->out_dtype == REPQ_BF16, REPQ_INVALID_ARG, "block_forward_host: bad out_dtype");
  if (n_batches == 0) return REPQ_OK;
  for (int k = 0; k < kSlots; ++k)
    REPQ_REQUIRE(s->x_dev[k] && s->y_dev[k], REPQ_INVALID_ARG, "block_forward_host: NULL staging buffer");
  REPQ_REQUIRE(s->x_dev[0] != s->x_dev[1] && s->y_dev[0] != s->y_dev[1], REPQ_INVALID_ARG,
               "block_forward_host: the two staging buffers of a direction must differ");
  for (int i = 0; i < n_batches; ++i)
    REPQ_REQUIRE(x_host[i] && y_host[i], REPQ_INVALID_ARG, "block_forward_host: NULL host buffer of batch %d", i);
  REPQ_REQUIRE(d->batch > 0 && d->seq > 0 && d->dim > 0, REPQ_INVALID_ARG, "block_forward_host: sizes must be positive");
  const size_t elems = size_t(d->batch) * size_t(d->seq) * size_t(d->dim);
  const size_t x_bytes = elems * dtype_size(d->act_dtype), y_bytes = elems * dtype_size(d->out_dtype);
  Pipeline* P = nullptr;
  REPQ_TRY(pipeline(&P));
  std::lock_guard<std::mutex> queueing(P->queueing);
  cudaStream_t main = static_cast<cudaStream_t>(stream);

  // the helper streams start after everything already queued on the caller's stream
  REPQ_CUDA(cudaEventRecord(P->start, main));
  REPQ_CUDA(cudaStreamWaitEvent(P->in, P->start, 0));
  REPQ_CUDA(cudaStreamWaitEvent(P->out, P->start, 0));
  const int pieces = pieces_of(x_bytes, *d, n_batches);
  const size_t x_item = x_bytes / size_t(d->batch), y_item = y_bytes / size_t(d->batch);
  auto first_item = [&](int c) { return size_t(int64_t(d->batch) * c / pieces); };
  // copy out of piece c of batch i, behind the copy in that `with` marks
  auto copy_out = [&](int i, int c, cudaEvent_t with) -> repq_status {
    const size_t first = first_item(c), bytes = (first_item(c + 1) - first) * y_item;
    const int k = i % kSlots;
    REPQ_CUDA(cudaStreamWaitEvent(P->out, P->computed[k][c], 0));
    if (with != nullptr && n_batches > 1) REPQ_CUDA(cudaStreamWaitEvent(P->out, with, 0));
    REPQ_CUDA(cudaMemcpyAsync(static_cast<uint8_t*>(y_host[i]) + first * y_item, static_cast<const uint8_t*>(s->y_dev[k]) + first * y_item, bytes,
                              cudaMemcpyDeviceToHost, P->out));
    REPQ_CUDA(cudaEventRecord(P->copied_out[k][c], P->out));
    return REPQ_OK;
  };
  repq_block_desc piece = *d;
  for (int i = 0; i < n_batches; ++i) {
    const int k = i % kSlots;
    for (int c = 0; c < pieces; ++c) {
      const size_t first = first_item(c), end = first_item(c + 1);
      piece.batch = int32_t(end - first);
      uint8_t* xd = static_cast<uint8_t*>(s->x_dev[k]) + first * x_item;
      uint8_t* yd = static_cast<uint8_t*>(s->y_dev[k]) + first * y_item;
      // copy in: this part of x_dev[k] was last read by the same piece of batch i - 2
      if (i >= kSlots) REPQ_CUDA(cudaStreamWaitEvent(P->in, P->computed[k][c], 0));
      REPQ_CUDA(cudaMemcpyAsync(xd, static_cast<const uint8_t*>(x_host[i]) + first * x_item, (end - first) * x_item, cudaMemcpyHostToDevice, P->in));
      REPQ_CUDA(cudaEventRecord(P->copied_in[k][c], P->in));
      // block: this part of y_dev[k] was last read by the copy-out of the same piece of batch i - 2
      REPQ_CUDA(cudaStreamWaitEvent(main, P->copied_in[k][c], 0));
      if (i >= kSlots) REPQ_CUDA(cudaStreamWaitEvent(main, P->copied_out[k][c], 0));
      REPQ_TRY(repq_block_forward(&piece, p, xd, yd, s->workspace, s->workspace_bytes, stream));
      REPQ_CUDA(cudaEventRecord(P->computed[k][c], main));
      // the piece before this one leaves with the next copy in
      if (c > 0) REPQ_TRY(copy_out(i, c - 1, P->copied_in[k][c]));
      else if (i > 0) REPQ_TRY(copy_out(i - 1, pieces - 1, P->copied_in[k][c]));
    }
  }
  REPQ_TRY(copy_out(n_batches - 1, pieces - 1, nullptr));
  // the caller's stream completes only after the last copy out (and hence, copies leaving in order, after every copy)
  REPQ_CUDA(cudaStreamWaitEvent(main, P->copied_out[(n_batches - 1) % kSlots][pieces - 1], 0));
  return REPQ_OK;
}
