// gen_resident_c.cu — instantiations of the resident generation kernel (rosenbrock, griewank).
#include "gen_resident.cuh"

namespace de {

const void* resident_entry_rosenbrock(bool seg, int vidx) { return resident_entry_obj<kRosenbrock>(seg, vidx); }
const void* resident_entry_griewank(bool seg, int vidx) { return resident_entry_obj<kGriewank>(seg, vidx); }

}  // namespace de
