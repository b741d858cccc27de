/* Layout 10 on tiles for one storage format and one high-order set size (one translation
 * unit each, so that they compile in parallel). */
#include "lb_tile.cuh"

namespace lbk {
template int launch_tiles_store<1, 36>(const StepParams<float> &, const RingTab &, const TileMaps &, const int4 *, int, int,
                                       uint32_t *, int *, void *);
}
