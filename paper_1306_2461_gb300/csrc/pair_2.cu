// Launches of one pair for window radius 2.
#define OF_RADIUS 2
#define OF_PAIR
#include "radius_impl.cuh"
