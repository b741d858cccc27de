/* Resident steps for one storage format and arithmetic (one translation unit each, so
 * that they compile in parallel). */
#include "lb_resident.cuh"

namespace lbk {
template int launch_resident_store<4, false>(const ResLaunch &);
}
