// tmem_share.h -- how the tensor-core kernels keep the CTAs that share an SM
// within its 512 columns of tensor memory. tcgen05.alloc waits, without a limit,
// until its columns are free, so every CTA also takes at least the same share of
// the SM's shared memory: CTAs that fit there together, of one kernel or of several
// that run at the same time (the weight gradients run beside the convolutions, and
// several networks beside one another), hold at most 512 columns.
#pragma once
#include <cstddef>
#include <cstdint>

namespace unet {

constexpr size_t kSmemMax = 227 * 1024;       // largest dynamic allocation of a CTA
constexpr size_t kSmemPerSM = 228 * 1024;
constexpr size_t kSmemReserved = 1024;        // taken by the system from every CTA's share
constexpr uint32_t kTmemColumns = 512;

// Dynamic shared memory of a CTA that needs `need` bytes and holds `cols` columns
// (0 < cols <= 512; 512 columns: 227 KB, 256: 113, 128: 56, as many CTAs an SM
// as its columns alone would allow).
constexpr size_t smem_floor(size_t need, uint32_t cols) {
  const size_t share = (kSmemPerSM * cols + kTmemColumns - 1) / kTmemColumns - kSmemReserved;
  return need > share ? need : share;
}

}  // namespace unet
