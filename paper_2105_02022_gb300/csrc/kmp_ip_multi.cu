// The bipartitioner's item kernel for graphs whose rows may hold parallel entries: the
// same source as kmp_ip.cu, with atomic updates of FM's keys and gains.
#define KMP_IP_MULTI 1
#include "kmp_ip.cu"
