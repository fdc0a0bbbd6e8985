// gen_resident_a.cu — instantiations of the resident generation kernel (sphere, rastrigin).
#include "gen_resident.cuh"

namespace de {

const void* resident_entry_sphere(bool seg, int vidx) { return resident_entry_obj<kSphere>(seg, vidx); }
const void* resident_entry_rastrigin(bool seg, int vidx) { return resident_entry_obj<kRastrigin>(seg, vidx); }

}  // namespace de
