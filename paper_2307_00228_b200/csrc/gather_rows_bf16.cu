#include "gather_rows.cuh"

it_status it_launch_gather_rows_bf16(const it_gather_args &a, const it_stream::StreamParams &sp, bool *folded, cudaStream_t st) { return launch_lpr<__nv_bfloat16>(a, sp, folded, st); }
