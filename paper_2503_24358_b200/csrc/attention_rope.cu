// Instances of the reader's kernel (attention_mma.cuh) for keys stored before the rotary embedding.
#include "attention_mma.cuh"

int squat_launch_attn_rope(const AttnParams &p, int bits, cudaStream_t st)
{
    return bits == 2 ? launch_q<true, 2>(p, st) : launch_q<true, 4>(p, st);
}
