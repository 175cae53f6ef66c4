// Launches of one pair for window radius 15.
#define OF_RADIUS 15
#define OF_PAIR
#include "radius_impl.cuh"
