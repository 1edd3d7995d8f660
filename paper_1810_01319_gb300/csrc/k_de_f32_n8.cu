// Float32 dual-energy sweeps of 8^3-cell blocks.
#define CELLO_DE_NB 8
#include "sweep_de_f32.cuh"
