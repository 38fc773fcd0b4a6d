// Arrivals at a grid barrier, counted modulo 2^32: a resident run without a rebuild
// passes 2^32 arrivals after some millions of steps (912 blocks: 4.7 million).  Of
// blocks that wait at barrier `phase` the count is never further than the number
// of blocks from the goal, so the sign of the difference decides.
#pragma once

#ifdef __CUDACC__
#define ESPP_HD __host__ __device__
#else
#define ESPP_HD
#endif

namespace espp {

ESPP_HD inline unsigned int barrier_goal(unsigned int blocks, unsigned int phase) { return blocks * phase; }
ESPP_HD inline bool barrier_reached(unsigned int seen, unsigned int goal) { return (int)(seen - goal) >= 0; }

}  // namespace espp
