// The wave kernel k_wave for packed copies (8-bit value numbers, 16-bit column distances): one
// right-hand side.
#include "mpk_wave.cuh"

namespace mpk {
void *select_wave_dict(int mode, int m, bool a32, WaveSize *size) {
    size->set<ValDict>();
    if (m != 1) fail(MPK_ERR_UNSUPPORTED, "packed copies are for one right-hand side, not %d", m);
    return wave_fn<ValDict, 1>(mode, a32);
}
}  // namespace mpk
