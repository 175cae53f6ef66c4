// Batched launches for window radius 12.
#define OF_RADIUS 12
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
