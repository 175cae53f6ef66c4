// Launches of one pair for window radius 4.
#define OF_RADIUS 4
#define OF_PAIR
#include "radius_impl.cuh"
