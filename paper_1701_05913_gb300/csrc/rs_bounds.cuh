// Index rules of the streaming kernels that the host can run too: no CUDA
// headers, so that a CPU test compiles them and checks every case.
#pragma once

#ifdef __CUDACC__
#define RS_HD __host__ __device__ __forceinline__
#else
#define RS_HD inline
#endif

#define RS_NO_STEP 0x7fffffff

// The consumer's step from which chunk q of a unit may be copied into ring slot
// q mod nslots: the step after the last one of chunk q - nslots, which held the
// slot before.  A unit has nch chunks of `steps` steps; past the last one there
// is no such step, also when the ring has more slots than the unit has chunks.
RS_HD int rs_wave_chunk_step(int q, int nch, int nslots, int steps)
{
    return q >= nch ? RS_NO_STEP : q < nslots ? 0 : (q - nslots + 1) * steps;
}
