// Batched launches for window radius 7.
#define OF_RADIUS 7
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
