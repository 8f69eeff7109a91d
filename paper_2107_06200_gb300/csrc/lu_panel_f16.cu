// lu_outer_panel for __half storage.
#include "lu_panel.cuh"

namespace msir {
cudaError_t launch_panel_f16(const PanelArgs& a, int C, cudaStream_t st) { return launch_panel_t<__half>(a, C, st); }
}  // namespace msir
