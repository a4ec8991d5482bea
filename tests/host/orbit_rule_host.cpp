// The orbit's stopping rule on the host.
#include "orbit_rule.cuh"

extern "C" int again(float u1, float u2) { return emri::orbit_again(u1, u2); }
extern "C" int settled(float p2, float p, float last) { return emri::orbit_settled(p2, p, last); }
