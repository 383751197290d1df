// kern_find.cu -- instantiations and launchers of the line find.
#include "ght_find_line.cuh"

namespace ght {

cudaError_t launch_find_line(bool key_slots, const TableView &tv, const uint32_t *q, uint32_t *out, uint64_t n,
                             bool early_exit, const LaunchOpts &o, cudaStream_t s) {
  return key_slots ? launch_line_find<KeySlot>(tv, q, out, n, early_exit, o.count, o.blocks_per_sm, s)
                   : launch_line_find<PairSlot>(tv, q, out, n, early_exit, o.count, o.blocks_per_sm, s);
}

}  // namespace ght
