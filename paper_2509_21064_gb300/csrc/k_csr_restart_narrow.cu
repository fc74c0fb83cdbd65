// Restart-resident sparse runs with 16-bit entries (see csr_restart.cuh).
#define RST_NARROW true
#define RST_PICK pick_narrow
#include "csr_restart.cuh"
