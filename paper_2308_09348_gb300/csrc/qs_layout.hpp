// qs_layout.hpp -- dynamic shared memory of the kernels whose regions mix
// types, laid out by one function for the kernel and for its launch.  Plain
// C++: the layouts are checked on the CPU for every block and bin count.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define QS_LAYOUT __host__ __device__ __forceinline__
#else
#define QS_LAYOUT inline
#endif

namespace qs {

QS_LAYOUT size_t align16(size_t bytes) { return (bytes + 15) & ~(size_t)15; }

// k_batch: a shot's launch constants (params bytes), the cycle tables (cycle
// bytes) and the shot's phase table (table bytes), both read as float4, 0 for
// none; then what is read in words of 8 bytes: the reduction scratch (red bytes
// per warp), the tile's spectrum (hist bytes), the work item (16) and the
// smoothed spectrum's accumulators (smooth bytes).  (The scratch is nine
// doubles per warp: behind it an odd number of warps would leave the tables 8
// bytes off.)
struct BatchLayout {
  size_t cycle, table, red, hist, item, smooth, bytes;
};
QS_LAYOUT BatchLayout batch_layout(size_t params, size_t cycle, size_t table, int warps, size_t red,
                                   size_t hist, size_t smooth) {
  BatchLayout l;
  l.cycle = align16(params);
  l.table = l.cycle + cycle;
  l.red = l.table + align16(table);
  l.hist = l.red + (size_t)warps * red;
  l.item = l.hist + align16(hist);
  l.smooth = l.item + 16;
  l.bytes = l.smooth + align16(smooth);
  return l;
}

// k_photon: the phase table (table bytes), the photon table (0 for none), the
// bin energies (eps bytes), the partial spectra (part bytes per warp), the
// emitters staged by each warp (stage bytes per warp) and the threads' states
// (state bytes per warp; the last two 0 for none).  The emitters are float4,
// the partial spectra before them doubles: an odd number of warps and of bins
// would leave the emitters 8 bytes off.
struct PhotonLayout {
  size_t ptab, eps, part, stage, state, bytes;
};
QS_LAYOUT PhotonLayout photon_layout(size_t table, size_t ptab, size_t eps, int warps, size_t part,
                                     size_t stage, size_t state) {
  PhotonLayout l;
  const size_t spectra = (size_t)warps * part;
  l.ptab = align16(table);
  l.eps = l.ptab + ptab;
  l.part = l.eps + align16(eps);
  l.stage = l.part + (stage ? align16(spectra) : spectra);
  l.state = l.stage + (size_t)warps * stage;
  l.bytes = l.state + (size_t)warps * state;
  return l;
}

}  // namespace qs
