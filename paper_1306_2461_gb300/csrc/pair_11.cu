// Launches of one pair for window radius 11.
#define OF_RADIUS 11
#define OF_PAIR
#include "radius_impl.cuh"
