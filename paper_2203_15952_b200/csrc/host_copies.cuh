// Layers on activations in host memory: copy in, compute and copy out of different rows at the same time.
#pragma once
#include <cmath>
#include <mutex>

#include "aqt_common.cuh"

namespace aqt {

// Two side streams, one for each copy direction, and the events that tie them to a caller's stream.  Lanes are kept for
// the life of the process, at most kCopyLanes a device.  A lane serves one call at a time (`busy`, while that call
// enqueues).  It is handed out again only when its last call's work has finished on the device or to a call on the same
// stream, which runs behind that work anyway: so no call ever waits for the work of another stream.
constexpr int kCopyLanes = 4;
constexpr int kCopyMaxDevices = 64;
struct CopyLane {
  cudaStream_t in = nullptr, out = nullptr;
  cudaEvent_t order = nullptr;  // of every record / wait pair (a wait takes the record before it)
  cudaEvent_t done = nullptr;   // end of the last call's work
  cudaStream_t user = nullptr;  // stream of the last call
  bool made = false, busy = false;
};
struct CopyLanes {
  std::mutex mutex;
  CopyLane lanes[kCopyMaxDevices][kCopyLanes];
};
inline CopyLanes& copy_lanes() {
  static CopyLanes* all = new CopyLanes;  // never destroyed: the driver may be gone when static destructors run
  return *all;
}

inline bool make_copy_lane(CopyLane* l) {
  if (cudaStreamCreateWithFlags(&l->in, cudaStreamNonBlocking) == cudaSuccess) {
    if (cudaStreamCreateWithFlags(&l->out, cudaStreamNonBlocking) == cudaSuccess) {
      if (cudaEventCreateWithFlags(&l->order, cudaEventDisableTiming) == cudaSuccess) {
        if (cudaEventCreateWithFlags(&l->done, cudaEventDisableTiming) == cudaSuccess) return true;
        cudaEventDestroy(l->order);
      }
      cudaStreamDestroy(l->out);
    }
    cudaStreamDestroy(l->in);
  }
  (void)cudaGetLastError();
  return false;
}

// A lane of the current device for a call on `st`, or null if every lane still has another stream's work.  *alone: no
// other stream has host copies under way.
inline CopyLane* take_copy_lane(cudaStream_t st, bool* alone) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kCopyMaxDevices) return nullptr;
  CopyLanes& all = copy_lanes();
  std::lock_guard<std::mutex> guard(all.mutex);
  CopyLane *own = nullptr, *idle = nullptr, *unmade = nullptr;
  *alone = true;
  for (CopyLane& l : all.lanes[dev]) {
    if (!l.made) {
      unmade = &l;
    } else if (l.busy) {
      *alone = false;
    } else if (l.user == st) {
      own = &l;
    } else if (cudaEventQuery(l.done) == cudaSuccess) {
      idle = &l;
    } else {
      (void)cudaGetLastError();
      *alone = false;
    }
  }
  CopyLane* pick = own != nullptr ? own : idle;
  if (pick == nullptr && unmade != nullptr && make_copy_lane(unmade)) {
    unmade->made = true;
    pick = unmade;
  }
  if (pick == nullptr) {
    *alone = false;
    return nullptr;
  }
  pick->busy = true;
  pick->user = st;
  return pick;
}
inline void give_back_copy_lane(CopyLane* l) {
  std::lock_guard<std::mutex> guard(copy_lanes().mutex);
  l->busy = false;
}

// Queries of events and the making of streams are refused, and break the capture, while another thread captures in the
// global mode.  None of them touches a captured stream here.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The address at which kernels reach these bytes of pinned host memory (whose copies run beside the host and beside each
// other), or null.  Both ends are looked up: of a buffer that is registered only in part, a kernel must not touch the rest.
inline void* pinned_on_device(const void* p, size_t bytes) {
  cudaPointerAttributes a, b;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess ||
      cudaPointerGetAttributes(&b, reinterpret_cast<const uint8_t*>(p) + (bytes > 0 ? bytes - 1 : 0)) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  if (a.type != cudaMemoryTypeHost || b.type != cudaMemoryTypeHost || a.devicePointer == nullptr) return nullptr;
  const bool whole = reinterpret_cast<uint8_t*>(b.devicePointer) == reinterpret_cast<uint8_t*>(a.devicePointer) + (bytes > 0 ? bytes - 1 : 0);
  return whole ? a.devicePointer : nullptr;
}

// Below this many bytes a kernel reads its input over the bus itself: no copy to set up and to wait for.  A quantizer that
// reads every element once: 0.7 MB 61 -> 53 us the whole feed-forward pair, 2 MB 114 -> 105 (6 MB by itself: 124 us, 125
// by the copy engine).  The chain kernel's CTAs read every row sixteen times: 8 rows of 512 22 -> 17 us, 16 rows alike,
// 32 rows 24 -> 33.
constexpr size_t kReadInPlaceBytes = 2000000, kReadInPlaceBytesChain = 20000;

// Rows of one piece.  The two copy directions run side by side and the compute hides between them, so a call takes one
// direction's time and one piece more, but every border between pieces costs both directions 14-25 us while they are
// both busy (4-5 us alone): the number of pieces grows with the root of the size.  Feed-forward pair, us whole / in
// this many pieces: 1.4 MB each way 89 / 84-155, 3.1 MB 145 / 128 (2), 12 MB 489 / 416 (2), 26 MB 1012 / 779 (3), 52 MB
// 2022 / 1471 (4), 134 MB 5096 / 3350 (6).  (Copied by SMs instead, either direction: 621-949 us where the copy engines
// move 26 MB both ways at once in 530.)
inline int64_t copy_piece_rows(int64_t rows, size_t row_bytes) {
  const double mb = (double)rows * (double)row_bytes * 1e-6;
  if ((size_t)rows * row_bytes < kReadInPlaceBytes) return rows;
  int64_t pieces = (int64_t)(sqrt(mb / 2.5) + 0.5);
  if (pieces < 2) pieces = 2;
  if (pieces > 6) pieces = 6;
#ifdef AQT_TUNING
  if (const char* e = tuning_env("AQT_PIECES")) pieces = atoi(e);
#endif
  return pieces < 2 ? rows : (int64_t)round_up((size_t)ceil_div(rows, pieces), 128);
}

// x_host -> x_dev, compute(first row, rows), y_dev -> y_host, for all rows, on `st` (null host pointers: no such copy).
// The pieces' copies run on a lane's streams, forked from and joined to `st`; compute enqueues on `st`.  One pass over
// all rows where a piece would be too small, where the memory is not pinned, while `st` is being captured, and while
// another stream has such a call under way: the two calls' copies overlap as they are, and pieces only add borders
// (12 800 x 512 in both directions on two streams in turn: 586 us a call whole, 641 in pieces).
template <class Compute>
int run_between_host_copies(const float* x_host, float* x_dev, size_t x_row, const float* y_dev, float* y_host, size_t y_row,
                            int64_t rows, cudaStream_t st, bool by_rows, Compute compute) {
  const size_t x_bytes = x_host != nullptr ? x_row : 0, y_bytes = y_host != nullptr ? y_row : 0;
  const int64_t piece = by_rows ? copy_piece_rows(rows, x_bytes > y_bytes ? x_bytes : y_bytes) : rows;
  CopyLane* lane = nullptr;
  bool alone = false;
  if (piece < rows) {
    RelaxedCapture relaxed;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone &&
        (x_host == nullptr || pinned_on_device(x_host, (size_t)rows * x_row) != nullptr) &&
        (y_host == nullptr || pinned_on_device(y_host, (size_t)rows * y_row) != nullptr))
      lane = take_copy_lane(st, &alone);
    else
      (void)cudaGetLastError();
  }
  if (!alone) {
    cudaError_t e = cudaSuccess;
    int rc = AQT_OK;
    if (x_host != nullptr) e = cudaMemcpyAsync(x_dev, x_host, (size_t)rows * x_row, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) rc = compute((int64_t)0, rows);
    if (e == cudaSuccess && rc == AQT_OK && y_host != nullptr) e = cudaMemcpyAsync(y_host, y_dev, (size_t)rows * y_row, cudaMemcpyDeviceToHost, st);
    if (lane != nullptr) {
      const cudaError_t d = cudaEventRecord(lane->done, st);
      if (e == cudaSuccess) e = d;
      give_back_copy_lane(lane);
    }
    return rc != AQT_OK ? rc : (e == cudaSuccess ? AQT_OK : AQT_ERR_CUDA);
  }
  const auto order = [lane](cudaStream_t first, cudaStream_t then) {
    cudaError_t e = cudaEventRecord(lane->order, first);
    return e != cudaSuccess ? e : cudaStreamWaitEvent(then, lane->order, 0);
  };
  const auto copy_in = [&](int64_t r0) {
    const int64_t n = rows - r0 < piece ? rows - r0 : piece;
    return cudaMemcpyAsync(reinterpret_cast<uint8_t*>(x_dev) + (size_t)r0 * x_row, reinterpret_cast<const uint8_t*>(x_host) + (size_t)r0 * x_row,
                           (size_t)n * x_row, cudaMemcpyHostToDevice, lane->in);
  };
  cudaError_t e = cudaSuccess;
  int rc = AQT_OK;
  if (x_host != nullptr) e = order(st, lane->in);
  if (e == cudaSuccess && x_host != nullptr) e = copy_in(0);
  for (int64_t r0 = 0; r0 < rows && e == cudaSuccess && rc == AQT_OK; r0 += piece) {
    const int64_t n = rows - r0 < piece ? rows - r0 : piece;
    if (x_host != nullptr) {
      e = order(lane->in, st);
      if (e == cudaSuccess && r0 + piece < rows) e = copy_in(r0 + piece);  // the copies stay ahead of the launches
    }
    if (e == cudaSuccess) rc = compute(r0, n);
    if (e == cudaSuccess && rc == AQT_OK && y_host != nullptr) {
      e = order(st, lane->out);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(reinterpret_cast<uint8_t*>(y_host) + (size_t)r0 * y_row, reinterpret_cast<const uint8_t*>(y_dev) + (size_t)r0 * y_row,
                            (size_t)n * y_row, cudaMemcpyDeviceToHost, lane->out);
    }
  }
  // joined whatever happened: what was enqueued still reads and writes the caller's buffers
  cudaError_t j = order(lane->in, st);
  const cudaError_t j2 = order(lane->out, st), j3 = cudaEventRecord(lane->done, st);
  if (j == cudaSuccess) j = j2 != cudaSuccess ? j2 : j3;
  give_back_copy_lane(lane);
  if (rc != AQT_OK) return rc;
  return e == cudaSuccess && j == cudaSuccess ? AQT_OK : AQT_ERR_CUDA;
}

}  // namespace aqt
