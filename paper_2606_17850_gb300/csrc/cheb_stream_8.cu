#include "cheb_stream.cuh"

th_status cheb_stream_8(thermal_grid* g, const Dims& d, const StreamChunk& c, cudaStream_t s) {
  return st_chunk<8>(g, d, c, s);
}
