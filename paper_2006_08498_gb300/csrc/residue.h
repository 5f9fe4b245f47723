// Shared between the residue products (residue.cu) and the product batcher
// (ozaki.cu): the jobs of one launch of k_res_zgemm.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

// One product C = A B in residues.  Its work units (column tile x row tile x
// K split x modulus) are numbered from unit0 on.
struct RsJob {
    CUtensorMap tmB;       // operand residues, box 64 x w
    const uint8_t *A;      // residues of A: [modulus][row tile][chunk][16 KB]
    uchar2 *R;             // residues of C + 128: [modulus][split][column < mp][row < Mp]
    ChaseScalars *sc;
    uint64_t wait_ns;      // limit of each bounded mbarrier wait
    int64_t Mp;            // rows, padded to whole row tiles
    int w, mp;             // columns of a column tile (a multiple of 16), of all tiles
    int nch, cs;           // K chunks, and chunks of one split
    int tx, ty, tz, nmod;  // column tiles, row tiles, splits, moduli
    int unit0;
};
constexpr int kRsMaxJobs = 8;
struct RsBatch {
    RsJob job[kRsMaxJobs];
    int njobs, units;
    int stride, slots;     // columns of an accumulator, and stages of A, in tensor memory
};
// Whether a job takes the three-product form: only such jobs share a launch.
bool rs_gauss(const RsJob &j);
inline int rs_units(const RsJob &j) { return j.tx * j.ty * j.tz * j.nmod; }
// Run a job through the batcher; returns after `st` waits for its launch.
struct OzBatcher;
cudaError_t ozb_run_residue(OzBatcher *b, const RsJob &job, cudaStream_t st);
cudaError_t residue_launch(RsBatch &b, int sms, cudaStream_t st);

// cuTensorMapEncodeTiled of the CUDA driver API (null when it is missing).
typedef CUresult (*TensorMapEncode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                    const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                    const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
TensorMapEncode tensor_map_encode();
