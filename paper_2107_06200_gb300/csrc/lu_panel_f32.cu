// lu_outer_panel for float storage.
#include "lu_panel.cuh"

namespace msir {
cudaError_t launch_panel_f32(const PanelArgs& a, int C, cudaStream_t st) { return launch_panel_t<float>(a, C, st); }
}  // namespace msir
