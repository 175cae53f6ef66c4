// Batched launches for window radius 11.
#define OF_RADIUS 11
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
