// instances.cuh -- the heavy kernels' instances of one shape order R, so that
// each order compiles in a translation unit of its own (instances_<R>.cu) and
// emu.cu only declares them (X empty here, extern there).
#pragma once

#include "kernels.cuh"
#include "kernels3d.cuh"
#include "kernels_general.cuh"

#define EMU_RK_STAGE(X, POT, R, S, TILES)                                                                           \
  X template __global__ void k_rk_stage<POT, R, S, TILES>(Batch, Parts, const double*, const double*,               \
                                                          const double*, const int*, const double*, const double*,  \
                                                          int, int);
#define EMU_RK_OTHER(X, POT, R, S)                                                                                  \
  X template __global__ void k3_rk_stage<POT, R, S>(Box3, Parts, double*, double*, const double*, const int*,       \
                                                    Field3, const int2*, int, int);                                 \
  X template __global__ void k_grk_stage<POT, R, S>(Batch, Parts, const int2*, const int2*, int, int);
#define EMU_RK_DEPOSIT(X, POT, R, S)                                                                                \
  X template __global__ void k_rk_deposit<POT, R, S>(Batch, Parts, double*, const double*, const int*,              \
                                                     const double*, int, double*, int*);
#define EMU_DEPOSIT(X, MODE, R, TAB, PART)                                                                                \
  X template __global__ void k_deposit<MODE, R, TAB, PART>(Batch, const double*, const double*, const double*,            \
                                                     const double*, const double*, const double*, const int*,       \
                                                     const double*, double, double*, double*, int*);
#define EMU_DEPOSIT_CLUSTER(X, R, TAB, CL)                                                                          \
  X template __global__ void k_deposit_cluster<R, TAB, CL>(Batch, const double*, const double*, const double*,      \
                                                           const double*, const double*, const double*, const int*, \
                                                           const double*, double, double*, double*, int*);
#define EMU_POT_INSTANCES(X, POT, R)                                                                                \
  EMU_RK_STAGE(X, POT, R, 1, 1)                                                                                     \
  EMU_RK_STAGE(X, POT, R, 2, 1)                                                                                     \
  EMU_RK_STAGE(X, POT, R, 4, 1)                                                                                     \
  EMU_RK_STAGE(X, POT, R, 1, kSlabTiles)                                                                            \
  EMU_RK_STAGE(X, POT, R, 2, kSlabTiles)                                                                            \
  EMU_RK_STAGE(X, POT, R, 4, kSlabTiles)                                                                            \
  X template __global__ void k_step<POT, R>(Batch, Parts, StepArgs);                                                \
  EMU_RK_OTHER(X, POT, R, 1)                                                                                        \
  EMU_RK_OTHER(X, POT, R, 2)                                                                                        \
  EMU_RK_OTHER(X, POT, R, 4)
#define EMU_ORDER_INSTANCES(X, R)                                                                                   \
  EMU_POT_INSTANCES(X, false, R)                                                                                    \
  EMU_POT_INSTANCES(X, true, R)                                                                                     \
  EMU_DEPOSIT(X, 0, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 1, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 2, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 3, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 3, R, false, true)                                                                                 \
  EMU_DEPOSIT(X, 3, R, true, false)                                                                                 \
  EMU_DEPOSIT(X, 3, R, true, true)                                                                                  \
  EMU_DEPOSIT(X, 4, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 5, R, false, false)                                                                                \
  EMU_DEPOSIT(X, 5, R, false, true)                                                                                 \
  EMU_DEPOSIT(X, 5, R, true, false)                                                                                 \
  EMU_DEPOSIT(X, 5, R, true, true)                                                                                  \
  EMU_DEPOSIT_CLUSTER(X, R, false, 8)                                                                               \
  EMU_DEPOSIT_CLUSTER(X, R, true, 8)                                                                                \
  EMU_DEPOSIT_CLUSTER(X, R, false, 16)                                                                              \
  EMU_DEPOSIT_CLUSTER(X, R, true, 16)
// Step form 2 (shape orders 0-2).
#define EMU_RD_INSTANCES(X, R)                                                                                      \
  EMU_RK_DEPOSIT(X, false, R, 0)                                                                                    \
  EMU_RK_DEPOSIT(X, false, R, 1)                                                                                    \
  EMU_RK_DEPOSIT(X, false, R, 2)                                                                                    \
  EMU_RK_DEPOSIT(X, false, R, 3)                                                                                    \
  EMU_RK_DEPOSIT(X, false, R, 4)                                                                                    \
  EMU_RK_DEPOSIT(X, true, R, 1)                                                                                     \
  EMU_RK_DEPOSIT(X, true, R, 2)                                                                                     \
  EMU_RK_DEPOSIT(X, true, R, 3)                                                                                     \
  EMU_RK_DEPOSIT(X, true, R, 4)
