// int16 with both cells (half codes, and larger codes): the queue's sweep kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_QUEUE_INSTANCE(5)
