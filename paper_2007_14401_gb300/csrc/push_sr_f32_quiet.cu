// push_sr_f32_quiet.cu -- push_sr_f32.cu without statistics (see GCB_STATS in push_sr.cuh).
#define GCB_STATS 0
#define GCB_FN(name) name##_quiet
#include "push_sr_f32.cu"
