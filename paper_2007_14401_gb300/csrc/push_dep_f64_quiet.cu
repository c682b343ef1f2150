// push_dep_f64_quiet.cu -- push_dep_f64.cu without statistics (see GCB_STATS in push_sr.cuh).
#define GCB_STATS 0
#define GCB_FN(name) name##_quiet
#include "push_dep_f64.cu"
