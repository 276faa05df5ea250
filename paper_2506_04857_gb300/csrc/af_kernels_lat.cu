// af_kernels_lat.cu -- the stage kernels of af_stage.cuh compiled for small grids.
#define AF_LAT 1
#include "af_stage.cuh"

void af_lat_pointdata(const AfDev &d, const AfGrid &g, int reduce_dt, cudaStream_t s) { launch_pointdata(d, g, reduce_dt, s); }
void af_lat_points(const AfDev &d, const AfGrid &g, double a, double b, int mode, cudaStream_t s) {
  launch_points(d, g, a, b, mode, s);
}
void af_lat_faces(const AfDev &d, const AfGrid &g, int mode, cudaStream_t s) { launch_faces(d, g, mode, s); }
void af_lat_cells(const AfDev &d, const AfGrid &g, double a, double b, int mode, cudaStream_t s) {
  launch_cells(d, g, a, b, mode, s);
}
void af_lat_final(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) { launch_final(d, g, a, b, s); }
void af_lat_lists(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) { launch_lists(d, g, a, b, s); }

#include "af_kernels1d.cuh"
