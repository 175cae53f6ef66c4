// Batched launches for window radius 16.
#define OF_RADIUS 16
#define OF_RADIUS_MORE
#include "radius_impl.cuh"
