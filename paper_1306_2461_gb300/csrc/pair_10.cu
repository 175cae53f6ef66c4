// Launches of one pair for window radius 10.
#define OF_RADIUS 10
#define OF_PAIR
#include "radius_impl.cuh"
