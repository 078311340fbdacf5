// Resident-trajectory tiles for BF16 rows of 41 to 64 covariates (tiles 24 and 25 of the table in
// res_bf16.cu). A translation unit of its own so that the library's
// sources compile in parallel.
#include "resident_wide.cuh"

namespace subsmc {

int res_launch_bf16_wide(int tile, const EstArgs &a, cudaStream_t s, int sms, bool dry) {
  switch (tile) {
    case 24: return launch_wide<7, 8>(a, s, sms, dry);
    case 25: return launch_wide<8, 8>(a, s, sms, dry);
    default: return -1;
  }
}

int res_launch_batch_bf16_wide(int tile, const BatchArgs &b, int p_max, int m_max, int G_max,
                               cudaStream_t s, int sms, bool dry) {
  switch (tile) {
    case 24: return launch_wide_batch<7, 8>(b, p_max, m_max, G_max, s, sms, dry);
    case 25: return launch_wide_batch<8, 8>(b, p_max, m_max, G_max, s, sms, dry);
    default: return -1;
  }
}

}  // namespace subsmc
