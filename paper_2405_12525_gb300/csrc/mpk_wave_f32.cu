// The wave kernel k_wave for matrix values stored as float32.
#include "mpk_wave.cuh"

namespace mpk {
void *select_wave_f32(int mode, int m, bool a32, WaveSize *size) { return select_wave_vt<ValF32>(mode, m, a32, size); }
}  // namespace mpk
