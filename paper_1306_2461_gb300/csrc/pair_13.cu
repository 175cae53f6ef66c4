// Launches of one pair for window radius 13.
#define OF_RADIUS 13
#define OF_PAIR
#include "radius_impl.cuh"
