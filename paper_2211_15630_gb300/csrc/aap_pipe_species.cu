// aap_pipe_species.cu -- the pipelined step kernel (aap_pipe.cu) for systems of
// several species (Sec. 2.5), a translation unit of its own so that the two
// compile side by side.  Three species, Langevin, N = 50,021 (400 tiles):
// 2310 us per 50 steps and state with the whole-block kernel it replaces there.
#define AAP_PIPE_SPECIES 1
#include "aap_pipe.cu"
