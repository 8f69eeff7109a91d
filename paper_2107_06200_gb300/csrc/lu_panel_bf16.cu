// lu_outer_panel for __nv_bfloat16 storage.
#include "lu_panel.cuh"

namespace msir {
cudaError_t launch_panel_bf16(const PanelArgs& a, int C, cudaStream_t st) { return launch_panel_t<__nv_bfloat16>(a, C, st); }
}  // namespace msir
