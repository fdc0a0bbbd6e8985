// gen_resident_b.cu — instantiations of the resident generation kernel (ackley, elliptic).
#include "gen_resident.cuh"

namespace de {

const void* resident_entry_ackley(bool seg, int vidx) { return resident_entry_obj<kAckley>(seg, vidx); }
const void* resident_entry_elliptic(bool seg, int vidx) { return resident_entry_obj<kElliptic>(seg, vidx); }

}  // namespace de
