// search_global.cu -- the layout optimiser (search.cuh) on layers too large for the shared memory of 16
// blocks (above about 60,000 neurons on 8 devices, 220,000 on 2): gains in the workspace.
#include "search.cuh"

namespace dtp {
namespace search {

Kernels kernels_in_global(int D) { return kernels_for<false>(D); }

}  // namespace search
}  // namespace dtp
