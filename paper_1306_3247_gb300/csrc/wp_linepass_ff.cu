// Passes over 512- to 2048-point lines held in registers for the float-float form.
#include <mutex>

#include "wp_linepass.cuh"

WP_LINEPASS_TU(ff)
