// Settings of the complex64 product that autotune.py chose over the defaults in
// matvec_kernels.cuh and fft_reg.cuh; at present the defaults stand.
#pragma once
