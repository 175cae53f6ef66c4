// Launches of one pair for window radius 5.
#define OF_RADIUS 5
#define OF_PAIR
#include "radius_impl.cuh"
