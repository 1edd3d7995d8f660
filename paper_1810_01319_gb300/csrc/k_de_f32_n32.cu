// Float32 dual-energy sweeps of 32^3-cell blocks.
#define CELLO_DE_NB 32
#include "sweep_de_f32.cuh"
