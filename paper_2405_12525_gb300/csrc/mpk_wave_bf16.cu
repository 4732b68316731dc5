// The wave kernel k_wave for matrix values stored as bfloat16.
#include "mpk_wave.cuh"

namespace mpk {
void *select_wave_bf16(int mode, int m, bool a32, WaveSize *size) { return select_wave_vt<ValBF16>(mode, m, a32, size); }
}  // namespace mpk
