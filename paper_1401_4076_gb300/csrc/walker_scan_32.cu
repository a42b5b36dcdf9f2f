// Walker update with several commits per round, 32 lanes per walker.
#include "walker_scan.cuh"

namespace mucal {

void walker_scan_32_fns(const void *(&fns)[kWalkerScanFns]) { walker_scan_fns_t<32>(fns); }

}  // namespace mucal
