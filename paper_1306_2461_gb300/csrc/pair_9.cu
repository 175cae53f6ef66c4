// Launches of one pair for window radius 9.
#define OF_RADIUS 9
#define OF_PAIR
#include "radius_impl.cuh"
