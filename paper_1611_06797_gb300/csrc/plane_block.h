// Thread block of the FP64 plane kernel (planes3_body_fx), host arithmetic only.
#pragma once

namespace ltmp2 {

struct PlaneBlock {
  int ib, threads;
};

// ib occupied planes of n x n points: a thread per line of their x pass, at most 256 threads (the kernel
// holds up to 255 registers), in whole warps: the plane's fixed-point scale comes from a sum over every
// lane of every warp, and in a warp that was launched in part the sum would read lanes that do not
// exist.  Idle threads cost nothing, the loops over the lines are strided.
inline PlaneBlock plane_block_f64(int n, int ib) {
  if (ib > 256 / n) ib = 256 / n;
  int threads = (ib * n + 31) / 32 * 32;
  if (threads < 64) threads = 64;
  return {ib, threads};
}

}  // namespace ltmp2
