// fpt_steps.h -- a trajectory's step count against its step cap.
//
// A lane counts groups of four steps; caps go up to 2^31 - 1 (the natural "no
// cap"), so 4 (groups + interval) does not fit an int near it. Every comparison
// is therefore made in groups. grp: groups taken by a live lane (4 grp <= nmax),
// groups: groups of the interval ahead.
#pragma once

#ifdef __CUDACC__
#define FPT_STEPS_FN __host__ __device__ __forceinline__
#else
#define FPT_STEPS_FN inline
#endif

namespace fpt_dev {

// Steps taken (modulo 2^32 for a lane without a trajectory, whose count is never read).
FPT_STEPS_FN int steps_of(int grp) { return (int)(4u * (unsigned)grp); }

// 4 (grp + groups) > nmax: the cap lies inside the interval.
FPT_STEPS_FN bool cap_inside(int grp, int groups, int nmax) { return grp > (nmax >> 2) - groups; }

// 4 grp >= nmax: the cap is reached.
FPT_STEPS_FN bool cap_reached(int grp, int nmax) { return grp > ((nmax - 1) >> 2); }

// 4 grp + 4 >= nmax: the cap is reached by the end of the next group.
FPT_STEPS_FN bool cap_in_group(int grp, int nmax) { return grp >= ((nmax - 1) >> 2); }

// 4 grp + k + 1 <= nmax: the group's step k (from 0) is within the cap.
FPT_STEPS_FN bool step_within(int grp, int k, int nmax) { return k < nmax - steps_of(grp); }

}  // namespace fpt_dev
