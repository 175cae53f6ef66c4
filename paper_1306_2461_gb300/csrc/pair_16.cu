// Launches of one pair for window radius 16.
#define OF_RADIUS 16
#define OF_PAIR
#include "radius_impl.cuh"
