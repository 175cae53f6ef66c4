// Launches of one pair for window radius 3.
#define OF_RADIUS 3
#define OF_PAIR
#include "radius_impl.cuh"
