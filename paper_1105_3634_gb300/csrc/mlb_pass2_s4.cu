// mlb_pass2_s4.cu -- pass 2 for four species (mlb_pass2.cuh).
#include "mlb_pass2.cuh"

MLBI_PASS2_UNIT(4)
