// Launches of one pair for window radius 7.
#define OF_RADIUS 7
#define OF_PAIR
#include "radius_impl.cuh"
