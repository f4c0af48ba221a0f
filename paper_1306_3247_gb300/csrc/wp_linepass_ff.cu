// Passes over 512- and 1024-point lines held in registers for the float-float form.
#include <mutex>

#include "wp_linepass.cuh"

WP_LINEPASS_TU(ff)
