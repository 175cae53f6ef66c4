// Launches of one pair for window radius 12.
#define OF_RADIUS 12
#define OF_PAIR
#include "radius_impl.cuh"
