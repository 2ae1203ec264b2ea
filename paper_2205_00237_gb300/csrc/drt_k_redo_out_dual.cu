// drt_k_redo_out_dual.cu -- the in-place redo with the rates the Doppler output needs (drt_k_redo_out.cu).
#define DRT_REDO_DUAL
#include "drt_k_redo_out.cu"
