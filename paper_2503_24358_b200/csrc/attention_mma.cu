// Instances of the reader's kernel (attention_mma.cuh) for keys stored after the rotary embedding.
#include "attention_mma.cuh"

int squat_launch_attn_mma(const AttnParams &p, int bits, cudaStream_t st)
{
    return bits == 2 ? launch_q<false, 2>(p, st) : launch_q<false, 4>(p, st);
}
