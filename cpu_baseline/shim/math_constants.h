// Host stand-in for the one CUDA math constant the binary64 solid code uses.
#pragma once
#define CUDART_INF (__builtin_inf())
// and the binary32 passes'
#define CUDART_INF_F (__builtin_inff())
