// What one CTA of a GEMM launch takes of its SM: shared memory and tensor-memory
// columns.  Plain host code, shared by the launches and by the CPU check of the
// rule below.
//
// Two kernels that run on the same SMs (two streams, two threads, or one kernel
// set up during another) may not both hold part of the tensor memory that a CTA
// pair waits for: tcgen05.alloc of a pair takes columns on both SMs, blocks without
// a limit, and nothing says that it takes them on both at once, so two pairs could
// each hold one SM's columns and wait for the other's.  CTAs of pairs therefore
// ask for at least kPairBytes + kPairColumnBytes x columns of shared memory: a pair
// has 64, 128, 256 or 512 columns, so CTAs that together exceed the 512 hold at
// least 576, and already two of them ask for more shared memory than an SM has
// (2 x 53,248 + 576 x 221 = 233,792 of 233,472 bytes).  Pairs that are resident
// together then have their columns at once.  One-SM CTAs need no rule: they wait
// for one SM's columns only, hold nothing meanwhile, and end without waiting for
// another CTA.
// The two constants leave the rings of 164 KB and more with 512 columns as they are
// (a GEMM alone takes the same time with any of them; what a larger one keeps out
// is the next preparation's blocks: 432 bytes for each column and nothing else
// made 4096 x 4096 x 1024 in 256 x 256 pair tiles with 3 stages, prepared and run,
// 43.3 -> 45.6 us).
#ifndef PM_FOOTPRINT_CUH
#define PM_FOOTPRINT_CUH

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace pm {

constexpr size_t kSmemPerSm = 233472;         // shared memory of an SM
constexpr size_t kSmemDynamic = 232448 - 1024;   // the most a GEMM CTA asks for (its barriers are static)
constexpr size_t kPairBytes = 53248, kPairColumnBytes = 221;

inline size_t pair_smem(size_t bytes, int columns) {
  return std::max(bytes, kPairBytes + kPairColumnBytes * (size_t)columns);
}

struct GemmFootprint {
  int acc_cols;          // columns of one accumulator buffer
  int a_cols;            // strategy B: columns of one stage's A copy
  int nbuf;              // accumulator buffers
  int alloc_cols;        // columns allocated
  uint32_t stage_bytes;  // one stage of the operand ring
  int staged;            // 4 KB staging buffers per epilogue warp: 2, 1 or 0
  size_t smem;           // dynamic shared memory of the launch
};

// Of a launch over G problems with tiles BM[q] x BN[q]; elem: bytes of an operand
// element, halves: operand planes (2 for three-pass TF32).
inline GemmFootprint gemm_footprint(int elem, int halves, int cg, int BK, int stages, int tmem_a, int G,
                                    const int16_t* BM, const int16_t* BN) {
  GemmFootprint f = {};
  int max_mblk = 1;
  for (int q = 0; q < G; ++q) {
    const int bm = BM[q], bn = BN[q], n_mblk = (bm + 127) / 128;
    f.acc_cols = std::max(f.acc_cols, (bm < 128 && cg == 2) ? bn / 2 : n_mblk * bn);
    max_mblk = std::max(max_mblk, n_mblk);
    f.stage_bytes = std::max(f.stage_bytes, (uint32_t)(halves * BK * elem) * (uint32_t)(bm + bn / cg));
  }
  // strategy B: one 8-column slot per 128-row x 32-byte A slice, per stage
  f.a_cols = tmem_a ? halves * (BK * elem / 4) * max_mblk : 0;
  const int a_ring = stages * f.a_cols;
  f.nbuf = (2 * f.acc_cols + a_ring <= 512) ? 2 : 1;
  f.alloc_cols = 32;
  while (f.alloc_cols < f.nbuf * f.acc_cols + a_ring) f.alloc_cols <<= 1;
  f.smem = (size_t)stages * f.stage_bytes + 1024;
  const size_t room = kSmemDynamic - f.smem;
  f.staged = room >= 32768 ? 2 : (room >= 16384 ? 1 : 0);
  f.smem += (size_t)f.staged * 16384;
  if (cg == 2) f.smem = pair_smem(f.smem, f.alloc_cols);
  return f;
}

}  // namespace pm

#endif  // PM_FOOTPRINT_CUH
