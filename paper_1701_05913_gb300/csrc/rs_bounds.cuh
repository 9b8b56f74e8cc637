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

// Sweeps of a part of nrow rows: places are 16 bits, idle records hold 0xFFFF.
// Once a copy has been given up on, RS_PART_LOST is in every place read, and the
// record, which is then whatever its ring slot held before, is not used.
#define RS_PART_LOST 0x10000
RS_HD bool rs_part_place(int e, int nrow) { return e < nrow; }
