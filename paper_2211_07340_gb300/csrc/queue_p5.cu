// int16 groups with codes too large for the half-code cell: the queue's sweep kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_QUEUE_INSTANCE(5)
