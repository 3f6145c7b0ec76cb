// Shape choices of the batched LU and the tensor-core routing thresholds on
// GB300 (hps_tune_set in include/hps.h), as paper_2503_17535_gb300/autotune.py writes
// them from timed builds of the benchmark workloads.  The base widths were then set
// from a sweep with the faster interchange step (few / many: 32/8, 64/16, 128/32,
// all/64 panels: 3D elliptic build 84.9 / 82.2 / 80.8 / 82.2 ms, Helmholtz 99.7 /
// 99.5 / 99.2 / 99.3); the work thresholds (2e5 .. 5e6) and the panel width (32; 24 and 16
// are slower) were swept again with the present kernels and stayed, the others are the
// autotuner's choice for earlier ones.
#pragma once

#define HPS_TUNED_LU_CLUSTER_PANEL 1
#define HPS_TUNED_LU_BASE_PANELS_FEW 128
#define HPS_TUNED_LU_FEW_MIN_N 4096
#define HPS_TUNED_LU_BASE_PANELS_MANY 32
#define HPS_TUNED_TC_MIN_WORK_REAL 50
#define HPS_TUNED_TC_MIN_WORK_CPLX 50
#define HPS_TUNED_TC_MIN_K 16
#define HPS_TUNED_TC_CHUNK_MB 1024
#define HPS_TUNED_TC_PERSIST_MIN_K 0
#define HPS_TUNED_LU_PANEL_NB_FEW 32
