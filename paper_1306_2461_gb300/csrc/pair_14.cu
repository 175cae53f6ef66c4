// Launches of one pair for window radius 14.
#define OF_RADIUS 14
#define OF_PAIR
#include "radius_impl.cuh"
