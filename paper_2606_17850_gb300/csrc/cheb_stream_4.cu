#include "cheb_stream.cuh"

th_status cheb_stream_4(thermal_grid* g, const Dims& d, const StreamChunk& c, cudaStream_t s) {
  return st_chunk<4>(g, d, c, s);
}
