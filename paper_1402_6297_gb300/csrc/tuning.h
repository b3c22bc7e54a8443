// Written by autotune.py: the complex64 product's kernel schedule for this GPU.
#pragma once
