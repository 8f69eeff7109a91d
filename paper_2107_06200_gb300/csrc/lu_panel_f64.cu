// lu_outer_panel for double storage.
#include "lu_panel.cuh"

namespace msir {
cudaError_t launch_panel_f64(const PanelArgs& a, int C, cudaStream_t st) { return launch_panel_t<double>(a, C, st); }
}  // namespace msir
