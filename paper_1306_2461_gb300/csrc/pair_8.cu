// Launches of one pair for window radius 8.
#define OF_RADIUS 8
#define OF_PAIR
#include "radius_impl.cuh"
