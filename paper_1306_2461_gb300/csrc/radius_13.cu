// Batched launches for window radius 13.
#define OF_RADIUS 13
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
