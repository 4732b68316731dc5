// The wave kernel k_wave for matrix values stored as float64.
#include "mpk_wave.cuh"

namespace mpk {
void *select_wave_f64(int mode, int m, bool a32, WaveSize *size) { return select_wave_vt<ValF64>(mode, m, a32, size); }
}  // namespace mpk
