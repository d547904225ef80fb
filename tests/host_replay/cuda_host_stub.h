// Host stand-ins for the CUDA qualifiers that csrc headers use.
#pragma once
#define __host__
#define __device__
#define __forceinline__ inline
