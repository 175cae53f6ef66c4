// Launches of one pair for window radius 0 (0: any radius, given at run time).
#define OF_RADIUS 0
#define OF_PAIR
#include "radius_impl.cuh"
