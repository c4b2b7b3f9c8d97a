// Lane capacity 32.
#define TSP_LMAX 32
#include "tsp_mlem_inst.cuh"
