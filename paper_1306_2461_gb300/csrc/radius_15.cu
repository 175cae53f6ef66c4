// Batched launches for window radius 15.
#define OF_RADIUS 15
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
