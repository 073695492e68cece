// The cluster form of the persistent time step (persist_shapes.cuh), in a translation unit of its own.
#include "persist_shapes.cuh"

namespace pncg {
PNCG_CLUSTER_DEF(float, false)
}
