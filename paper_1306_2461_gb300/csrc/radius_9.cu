// Batched launches for window radius 9.
#define OF_RADIUS 9
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
