// Float32 dual-energy sweeps of 16^3-cell blocks.
#define CELLO_DE_NB 16
#include "sweep_de_f32.cuh"
