// Batched launches for window radius 14.
#define OF_RADIUS 14
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
