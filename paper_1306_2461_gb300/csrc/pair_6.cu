// Launches of one pair for window radius 6.
#define OF_RADIUS 6
#define OF_PAIR
#include "radius_impl.cuh"
