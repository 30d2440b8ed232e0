// Internal launchers shared by the C-ABI entry points and the context.
#pragma once

#include "common.cuh"

struct rbfsl_knn_index {
    int device;
    int64_t N;
    int G;                 // cells per axis over [-1, 1]^3
    double cell;           // cell edge 2 / G
    double r2_per_k;       // initial squared search radius per neighbour: 4 * 1.3 / N
    double *sx, *sy, *sz;  // node coordinates sorted by cell (SoA)
    int32_t *sid;          // original node index of each sorted entry
    int32_t *cell_start;   // G^3 + 1 offsets into the sorted arrays
    size_t bytes;
};

// RBF-PU patches and factors (pu.cu).
struct rbfsl_pu {
    int device = 0;
    int64_t N = 0, Mp = 0;
    double R = 0;
    int ell = 0, power = 0, M = 0, max_members = 0;
    double *X = nullptr, *centers = nullptr;
    int64_t *mstart = nullptr;   // Mp + 1 (device)
    int32_t *members = nullptr;  // mstart[Mp] (device), ascending node index per patch
    int reduced = 0;             // 1: reduced factors as digits (PatchLayout), 0: LU factors
    int64_t *lu_off = nullptr;   // Mp (device): offset of patch l's factors
    double *LU = nullptr;
    int32_t *perm = nullptr;     // pivot (reduced) or row (LU) order, at mstart[l] + l * M
    int32_t *pmem = nullptr;     // reduced: members in pivot order, at mstart[l]
    double *mx = nullptr;        // members' coordinates, patch l's from row mstart[l] + l M on
    rbfsl_knn_index *nodes_ix = nullptr, *centers_ix = nullptr;
    void *coef = nullptr;        // (mstart[Mp] + Mp M) x coef_T values of 8 bytes at most
    int coef_T = 0;
    int64_t rows = 0;            // mstart[Mp] + Mp M
    int64_t chunk = 0;           // points per launch of the blend, and their patches and harmonics
    int32_t *pt_cnt = nullptr, *pt_id = nullptr;
    double *pt_w = nullptr, *pt_Y = nullptr;
    cudaStream_t side = nullptr;  // the coefficients, beside the tracing and the points' patches
    cudaEvent_t fork = nullptr, join = nullptr;
    int32_t *status = nullptr;
    size_t bytes = 0;
};

namespace rbfsl {

// Device view of a grid index (see knn.cu).
struct KnnGrid {
    const double *sx, *sy, *sz;
    const int32_t *sid, *cell_start;
    int G;
    double r2_per_k;
};

inline KnnGrid grid_view(const rbfsl_knn_index *ix) {
    return KnnGrid{ix->sx, ix->sy, ix->sz, ix->sid, ix->cell_start, ix->G, ix->r2_per_k};
}

__device__ __forceinline__ int cell_coord(double v, double inv_cell, int G) {
    int c = (int)floor((v + 1.0) * inv_cell);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

// Calls f(p, on) for the indexed points (sorted positions p, each once) of the cells that overlap the
// ball of radius rb around (qx, qy, qz), 32 at a time: the whole warp calls f, on = false in lanes
// without a point. The cells of a grid row (fixed y and z) are neighbours in the sorted order, so a
// row's part of the ball is one range; the lanes take a row each, narrow its x-extent to the ball's
// chord, and the ranges are dealt to the lanes point by point (a prefix sum of their lengths), so
// that lanes idle in the last 32 only. A cell to a lane, with the whole bounding box, left most
// lanes waiting for the few with occupied cells (k-NN, k = 84, N = 40,962: 984 us against 216 us).
// Row and chord tests in FP32 with margins that cover its rounding: cells are only added. Cells on
// the grid's border hold every point beyond it and are not narrowed on that side.
template <typename F>
__device__ __forceinline__ void grid_ball_foreach(const KnnGrid &g, double qx, double qy, double qz,
                                                  float rb, int lane, F f) {
    const float x = (float)qx, y = (float)qy, z = (float)qz, r = rb * 1.00001f + 1e-6f;
    const float inv = 0.5f * (float)g.G, edge = 1.0f / inv;
    const int G = g.G;
    auto cell = [&](float v, float margin) {
        const int c = (int)floorf((v + 1.0f) * inv + margin);
        return c < 0 ? 0 : (c >= G ? G - 1 : c);
    };
    auto outside = [&](float v, int c) {  // distance of v from cell c's interval
        const float lo = c == 0 ? -1e30f : c * edge - 1.0f, hi = c == G - 1 ? 1e30f : (c + 1) * edge - 1.0f;
        return fmaxf(fmaxf(lo - v, v - hi), 0.0f);
    };
    const int y0 = cell(y - r, -1e-3f), y1 = cell(y + r, 1e-3f), z0 = cell(z - r, -1e-3f), z1 = cell(z + r, 1e-3f);
    const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
    for (int base = 0; base < rows; base += 32) {
        int b = 0, cnt = 0;
        if (base + lane < rows) {
            const int q = (base + lane) / ny, cz = z0 + q, cy = y0 + (base + lane - q * ny);
            const float dy = outside(y, cy), dz = outside(z, cz);
            const float h2 = r * r - dy * dy - dz * dz;
            if (h2 >= -1e-4f * r * r) {
                const float h = sqrtf(fmaxf(h2, 0.0f)) * 1.00001f + 0.02f * r;
                const int64_t c = (int64_t)(cz * G + cy) * G;
                b = g.cell_start[c + cell(x - h, -1e-3f)];
                cnt = g.cell_start[c + cell(x + h, 1e-3f) + 1] - b;
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int i0 = 0; i0 < total; i0 += 32) {
            const int i = i0 + lane;
            int row = 0;  // the first range that ends behind i
#pragma unroll
            for (int st = 16; st > 0; st >>= 1)
                if (__shfl_sync(0xffffffffu, incl, row + st - 1) <= i) row += st;
            row = row > 31 ? 31 : row;
            const int p = __shfl_sync(0xffffffffu, b + cnt - incl, row) + i;
            f(p, i < total);
        }
    }
}

// The same for one thread: f(p) for the sorted positions p of the cells that the ball touches.
template <typename F>
__device__ __forceinline__ void grid_ball_rows(const KnnGrid &g, double qx, double qy, double qz, float rb, F f) {
    const float x = (float)qx, y = (float)qy, z = (float)qz, r = rb * 1.00001f + 1e-6f;
    const float inv = 0.5f * (float)g.G, edge = 1.0f / inv;
    const int G = g.G;
    auto cell = [&](float v, float margin) {
        const int c = (int)floorf((v + 1.0f) * inv + margin);
        return c < 0 ? 0 : (c >= G ? G - 1 : c);
    };
    auto outside = [&](float v, int c) {
        const float lo = c == 0 ? -1e30f : c * edge - 1.0f, hi = c == G - 1 ? 1e30f : (c + 1) * edge - 1.0f;
        return fmaxf(fmaxf(lo - v, v - hi), 0.0f);
    };
    const int y0 = cell(y - r, -1e-3f), y1 = cell(y + r, 1e-3f), z0 = cell(z - r, -1e-3f), z1 = cell(z + r, 1e-3f);
    // four rows' ranges are loaded together: a thread by itself waits for each of its loads
    const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
    int cy = y0, cz = z0;
    for (int base = 0; base < rows; base += 4) {
        int b[4], e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            b[u] = e[u] = 0;
            const float dy = outside(y, cy), dz = outside(z, cz), h2 = r * r - dy * dy - dz * dz;
            if (base + u < rows && h2 >= -1e-4f * r * r) {
                const float h = sqrtf(fmaxf(h2, 0.0f)) * 1.00001f + 0.02f * r;
                const int64_t c = (int64_t)(cz * G + cy) * G;
                b[u] = g.cell_start[c + cell(x - h, -1e-3f)];
                e[u] = g.cell_start[c + cell(x + h, 1e-3f) + 1];
            }
            if (++cy > y1) {
                cy = y0;
                ++cz;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            for (int p = b[u]; p < e[u]; ++p) f(p);
    }
}

int launch_trace(const double *x, int64_t N, int vel_kind, const double *prm, double t1,
                 double dt, int precision, double *xi, cudaStream_t s);

int knn_index_build(rbfsl_knn_index *ix, const double *x, int64_t N, int k_hint, cudaStream_t s);
void knn_index_free(rbfsl_knn_index *ix);
int launch_knn(const rbfsl_knn_index *ix, const double *q, int64_t Nq, int k, int32_t *idx,
               int32_t *status, cudaStream_t s);

int launch_weights(const double *x, const int32_t *idx, int64_t Nq, int n, int ell, int power,
                   const double *p, void *w, int w_dtype, int32_t *status, cudaStream_t s);

int launch_trace_order(const double *x, int64_t N, int vel_kind, const double *prm, double t1, double dt,
                       int precision, int order, double *xi, cudaStream_t s);

int launch_gather(const int32_t *idx, const void *w, int64_t Nq, int n, const void *q, int T,
                  int dtype, void *q_out, cudaStream_t s);

int sh_tables_init();

// rbfsl_pu_apply in two parts. begin: the coefficients of a field of q_dtype (RBFSL_F64, or RBFSL_F32X2: FP32
// pairs) on the handle's side stream, after what is on s; end (also after an error in between): the points'
// patches on s, then, with the coefficients there, the blend. q must stay unchanged until end's work on s.
int pu_apply_begin(rbfsl_pu *u, const void *q, int q_dtype, int T, int dtype, cudaStream_t s);
int pu_apply_end(rbfsl_pu *u, int T, const double *p, int64_t Nq, int wkind, int dtype, void *out, int32_t *status,
                 cudaStream_t s);

size_t pu_estimate_bytes(int64_t N, int64_t Mp, int members, int ell, int power, int T);

int launch_stencil_factor(const double *X, const int64_t *mstart, const int32_t *members,
                          const int64_t *lu_off, int64_t count, int max_n, int M, int ell,
                          int power, double *LU, int32_t *perm, int32_t *status, cudaStream_t s,
                          int colmajor);

// Kept factors of the centre stencils Ik (N x n): in the reduced form (reduced.cuh) or, where that
// does not serve the system or breaks down at a stencil, LU of the whole systems.
struct CenterFactors {
    double *F = nullptr;       // per stencil: CenterLayout, or m x m column-major LU
    int32_t *order = nullptr;  // per stencil: n (reduced) or m positions
    int reduced = 0;
    size_t bytes = 0;
};
int center_factors_build(const double *X, const int32_t *Ik, int64_t N, int n, int ell, int power,
                         CenterFactors *out, cudaStream_t s);
void center_factors_free(CenterFactors *f);
int launch_center_weights(const double *X, const int32_t *K, const int32_t *Ik, const CenterFactors &f, int64_t Nq,
                          int n, int ell, int power, const double *p, int32_t *I, void *w, int w_dtype,
                          int32_t *status, cudaStream_t s);

int global_factor_full(const double *x, int64_t N, int kernel, double eps, double *LU, int32_t *perm,
                       int32_t *piv, int32_t *status, cudaStream_t s);
int global_factor_chol_full(const double *x, int64_t N, int kernel, double eps, double *LU, int32_t *perm,
                            cudaStream_t s);
int global_solve(const double *LU, const int32_t *perm, int64_t N, const double *Q, int T,
                 double *C, cudaStream_t s);
int launch_global_eval(const double *P, int64_t Nq, const double *X, int64_t N, int kind,
                       double eps, const void *C, int T, int dtype, void *out, int out_dtype,
                       cudaStream_t s);
size_t global_eval_tc_workspace(int64_t Nq, int64_t N, int T);
int launch_global_eval_tc(const double *P, int64_t Nq, const double *X, int64_t N, int kind, double eps,
                          const void *C, int c_dtype, int T, float *out, void *workspace, int32_t *status,
                          cudaStream_t s);

int global_cardinal_build(const double *LU, const int32_t *perm, const double *X, int64_t N, int kind,
                          double eps, const double *P, int64_t Nq, void *E, int e_dtype, cudaStream_t s);
size_t cardinal_apply_workspace(int64_t Nq, int64_t N, int T);
int launch_cardinal_apply(const void *E, int64_t Nq, int64_t N, const void *q, int T, int dtype, void *out,
                          void *ws, size_t ws_bytes, cudaStream_t s);

}  // namespace rbfsl
