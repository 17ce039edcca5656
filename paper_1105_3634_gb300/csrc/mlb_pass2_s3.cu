// mlb_pass2_s3.cu -- pass 2 for three species (mlb_pass2.cuh).
#include "mlb_pass2.cuh"

MLBI_PASS2_UNIT(3)
