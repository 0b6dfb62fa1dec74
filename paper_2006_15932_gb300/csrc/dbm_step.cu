// dbm_step.cu -- dispatch of the fused step on precision, species count and
// kernel variant, and the TMA descriptors of the state buffers.  The
// kernels are in dbm_step_impl.cuh, instantiated once per species count in
// dbm_step_s<S>.cu so that the units compile in parallel.
#include <stdio.h>
#include <string.h>

#include "dbm_internal.h"

namespace dbm {

template <int S>
int launch_step_t(dbm_handle *h, const void *fin, void *fout, cudaStream_t st);
template <int S, int TX, int TY, int CW, int MODE>
int launch_step_tma_t(dbm_handle *h, const CUtensorMap *tmap, const CUtensorMap *tmap_in, const void *fin, void *fout,
                      cudaStream_t st);
template <int S, int TX, int TY>
int launch_step_half_t(dbm_handle *h, const CUtensorMap *tmap, const CUtensorMap *tmap_in, const void *fin, void *fout,
                       cudaStream_t st);
template <int S, int TX, int TY, int CW>
int launch_step_staged_t(dbm_handle *h, const CUtensorMap *tmap, const CUtensorMap *tmap_in, const void *fin,
                         void *fout, cudaStream_t st);

template <int S>
static int launch_staged_s(dbm_handle *h, const CUtensorMap *tm, const CUtensorMap *ti, const void *fin, void *fout,
                           cudaStream_t st)
{
    if constexpr (S >= 5)
        if (h->tma_cw == 1) return launch_step_staged_t<S, STAGED_TX, STAGED_TY, 1>(h, tm, ti, fin, fout, st);
    return launch_step_staged_t<S, PAIR_TX, PAIR_TY, 2>(h, tm, ti, fin, fout, st);
}

// The species-staged step of the handle's tile (no arithmetic options).
static int launch_staged(dbm_handle *h, int cur, const void *fin, void *fout, cudaStream_t st)
{
    const CUtensorMap *tm = &h->tmap[cur], *ti = &h->tmap_in[cur];
    switch (h->p.nspecies) {
    case 2: return launch_staged_s<2>(h, tm, ti, fin, fout, st);
    case 3: return launch_staged_s<3>(h, tm, ti, fin, fout, st);
    case 4: return launch_staged_s<4>(h, tm, ti, fin, fout, st);
    case 5: return launch_staged_s<5>(h, tm, ti, fin, fout, st);
    case 6: return launch_staged_s<6>(h, tm, ti, fin, fout, st);
    case 7: return launch_staged_s<7>(h, tm, ti, fin, fout, st);
    case 8: return launch_staged_s<8>(h, tm, ti, fin, fout, st);
    }
    return DBM_ERR_INVALID;
}

// The TMA-staged step of the handle's tile with the FP32 arithmetic options
// MODE (acc_mode).
template <int MODE>
static int launch_tma(dbm_handle *h, const CUtensorMap *tm, const CUtensorMap *ti, const void *fin, void *fout,
                      cudaStream_t st)
{
    if (h->tma_half)
        return h->p.nspecies == 2 ? launch_step_half_t<2, SMALL_TX, SMALL_TY>(h, tm, ti, fin, fout, st)
                                  : launch_step_half_t<4, SMALL_TX, SMALL_TY>(h, tm, ti, fin, fout, st);
    switch (h->p.nspecies) {
    case 1: return launch_step_tma_t<1, tma_tile_x(1), tma_tile_y(1), 1, MODE>(h, tm, ti, fin, fout, st);
    case 2:
        if (h->tma_cw == 2) return launch_step_tma_t<2, PAIR_TX, PAIR_TY, 2, MODE>(h, tm, ti, fin, fout, st);
        return launch_step_tma_t<2, tma_tile_x(2), tma_tile_y(2), 1, MODE>(h, tm, ti, fin, fout, st);
    case 3: return launch_step_tma_t<3, tma_tile_x(3), tma_tile_y(3), 1, MODE>(h, tm, ti, fin, fout, st);
    case 4: return launch_step_tma_t<4, tma_tile_x(4), tma_tile_y(4), 1, MODE>(h, tm, ti, fin, fout, st);
    }
    return DBM_ERR_INVALID;
}

// The all-species TMA-staged kernels exist for FP32 with up to four species;
// the species-staged one for two to eight species without the arithmetic
// options.
bool tma_supported(const dbm_params &p) { return p.precision == DBM_FP32 && p.nspecies <= 4; }
static bool staged_supported(const dbm_params &p)
{
    return p.precision == DBM_FP32 && p.nspecies >= 2 && p.nspecies <= DBM_MAX_SPECIES && !uses_acc(p);
}

static long long pair_tiles(const dbm_params &p)
{
    return (long long)((p.nx + PAIR_TX - 1) / PAIR_TX) * ((p.ny + PAIR_TY - 1) / PAIR_TY);
}

// The tile of the TMA-staged step, without the arithmetic options:
// two species: two threads per pair, whose chain is the shortest, while three
//   small tiles per SM hold the grid (us a step, two threads / pairs, on 152 SMs:
//   256 x 128 6.1 / 8.0, 256 x 200, 400 tiles, 6.3 / 8.1, 704 x 80, 440 tiles, 6.4 /
//   8.3; past 456 tiles a second wave: 832 x 72, 468, 9.3 / 8.3, 768 x 80, 480, 9.8 /
//   8.4), then two cells per thread (one cell / pairs: 4096^2 845 / 726, 1024^2
//   68 / 60, 1001 x 771 51 / 45, 512^2 20.0 / 17.7);
// one and three species: one cell per thread (three species, two threads per
//   pair: 128^2 7.5 / 8.0, 256^2 9.9 / 14.6; species-staged: 2048 x 1024 174 /
//   201);
// four: one cell per thread (2048 x 1024 261, species-staged 265), two threads
//   per pair on grids of at most one small tile per SM (one cell / two threads:
//   64^2 8.7 / 7.7, 128^2 8.4 / 8.1, 777 x 413 57 / 91);
// five or more: the species-staged kernel, the only TMA-staged one.
// DBM_KERNEL_TMA_CELL asks for one cell per thread, DBM_KERNEL_TMA_PAIR for two
// (three and more species: staged), DBM_KERNEL_TMA_STAGED for the
// species-staged kernel, in pairs up to four species and one cell per thread
// from five on.  With an option: two species pairs from PAIR_MIN_TILES
// tiles up, else one cell.
static void choose_tile(dbm_handle *h)
{
    const dbm_params &p = h->p;
    const int want = p.step_kernel;
    h->tma_staged = h->tma_half = 0;
    const bool staged_by_default = p.nspecies > 4 && want != DBM_KERNEL_TMA_CELL;
    const bool staged_asked = want == DBM_KERNEL_TMA_STAGED || (p.nspecies >= 3 && want == DBM_KERNEL_TMA_PAIR);
    if (staged_supported(p) && (staged_by_default || staged_asked)) {
        h->tma_staged = 1;
        const bool pair = p.nspecies < 5 || want == DBM_KERNEL_TMA_PAIR;
        h->tma_tx = pair ? PAIR_TX : STAGED_TX;
        h->tma_ty = pair ? PAIR_TY : STAGED_TY;
        h->tma_cw = pair ? 2 : 1;
        return;
    }
    const long long small = (long long)((p.nx + SMALL_TX - 1) / SMALL_TX) * ((p.ny + SMALL_TY - 1) / SMALL_TY);
    h->tma_half = !uses_acc(p) && want != DBM_KERNEL_TMA_CELL && want != DBM_KERNEL_TMA_PAIR &&
                  small <= (long long)small_tiles_per_sm(p.nspecies) * h->sms;
    const bool pair = p.nspecies == 2 && want != DBM_KERNEL_TMA_CELL && !h->tma_half &&
                      (want == DBM_KERNEL_TMA_PAIR || !uses_acc(p) || pair_tiles(p) >= PAIR_MIN_TILES);
    h->tma_tx = pair ? PAIR_TX : h->tma_half ? SMALL_TX : tma_tile_x(p.nspecies);
    h->tma_ty = pair ? PAIR_TY : h->tma_half ? SMALL_TY : tma_tile_y(p.nspecies);
    h->tma_cw = pair ? 2 : 1;
}

// dbm_step_tile's answer: a rule of its own, which programs have read and
// dbm.h states; the step follows choose_tile.
static void told_tile(dbm_handle *h)
{
    const dbm_params &p = h->p;
    const bool pair = h->tma_staged || (p.nspecies == 2 && p.step_kernel != DBM_KERNEL_TMA_CELL &&
                                        (p.step_kernel == DBM_KERNEL_TMA_PAIR || pair_tiles(p) >= PAIR_MIN_TILES));
    h->told_tx = pair ? PAIR_TX : tma_tile_x(p.nspecies);
    h->told_ty = pair ? PAIR_TY : p.nspecies == 4 ? 6 : tma_tile_y(p.nspecies);
    h->told_cw = pair ? 2 : 1;
}

int step_kernel_name(const dbm_handle *h, char *name, size_t size)
{
    const dbm_params &p = h->p;
    const int S = p.nspecies;
    if (p.precision == DBM_FP64) {
        snprintf(name, size, "%s<%d>", f64_small_grid(h) ? "k_step_f64_small" : "k_step_f64", S);
    } else if (p.precision == DBM_BF16DEV) {
        snprintf(name, size, "k_step_bf16<%d,%d,%d,%d>", S, BF_TX, BF_TY, BF_CW);
    } else if (!h->tma_ok || p.step_kernel == DBM_KERNEL_GENERIC) {
        if (uses_acc(p) || (p.step_kernel != DBM_KERNEL_AUTO && p.step_kernel != DBM_KERNEL_GENERIC))
            return DBM_ERR_INVALID;
        snprintf(name, size, "k_step<%d>", S);
    } else if (h->tma_half) {
        snprintf(name, size, "k_step_half<%d,%d,%d>", S, h->tma_tx, h->tma_ty);
    } else {
        snprintf(name, size, "%s<%d,%d,%d,%d>", h->tma_staged ? "k_step_staged" : "k_step_tma", S, h->tma_tx, h->tma_ty,
                 h->tma_cw);
    }
    return DBM_OK;
}

typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

// One 3-D descriptor per state buffer: (column, row, plane) with the whole
// padded geometry; out-of-range boxes are zero-filled by the copy engine.
int make_tensor_maps(dbm_handle *h)
{
    h->tma_ok = 0;
    h->tma_tx = h->tma_ty = h->tma_cw = h->tma_staged = 0;
    if (!tma_supported(h->p) && !staged_supported(h->p)) return DBM_OK;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return DBM_OK;  // no TMA descriptors: the generic kernel runs
    }
    encode_tiled_fn encode = (encode_tiled_fn)fn;
    const dbm_layout &L = h->lay;
    cuuint64_t dims[3] = {(cuuint64_t)L.pitch, (cuuint64_t)L.rows, (cuuint64_t)(16 * h->p.nspecies)};
    cuuint64_t strides[2] = {(cuuint64_t)L.pitch * 4, (cuuint64_t)L.plane * 4};
    choose_tile(h);
    told_tile(h);
    if (!h->tma_staged && !tma_supported(h->p)) {  // no all-species kernel for this species count
        h->tma_tx = h->tma_ty = h->tma_cw = 0;
        return DBM_OK;
    }
    // the box: the tile, its halo and one species' planes
    const cuuint32_t planes = (cuuint32_t)Q;
    cuuint32_t box[3] = {(cuuint32_t)(h->tma_tx + 8), (cuuint32_t)(h->tma_ty + 4), planes};
    cuuint32_t estr[3] = {1, 1, 1};
    for (int k = 0; k < 2; ++k) {
        CUresult r = encode(&h->tmap[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, h->f[k], dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r == CUDA_SUCCESS) {  // interior box of one species: the tile's own cells
            cuuint32_t box_in[3] = {(cuuint32_t)h->tma_tx, (cuuint32_t)h->tma_ty, (cuuint32_t)Q};
            r = encode(&h->tmap_in[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, h->f[k], dims, strides, box_in, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        }
        if (r != CUDA_SUCCESS) {
            h->tma_tx = h->tma_ty = h->tma_cw = h->tma_staged = 0;
            return DBM_OK;
        }
    }
    h->tma_ok = 1;
    return DBM_OK;
}

static int launch_generic(dbm_handle *h, const void *fin, void *fout, cudaStream_t st)
{
    switch (h->p.nspecies) {
    case 1: return launch_step_t<1>(h, fin, fout, st);
    case 2: return launch_step_t<2>(h, fin, fout, st);
    case 3: return launch_step_t<3>(h, fin, fout, st);
    case 4: return launch_step_t<4>(h, fin, fout, st);
    case 5: return launch_step_t<5>(h, fin, fout, st);
    case 6: return launch_step_t<6>(h, fin, fout, st);
    case 7: return launch_step_t<7>(h, fin, fout, st);
    case 8: return launch_step_t<8>(h, fin, fout, st);
    }
    return DBM_ERR_INVALID;
}

int launch_step(dbm_handle *h, int cur, cudaStream_t st)
{
    const void *fin = h->f[cur];
    void *fout = h->f[cur ^ 1];
    const int want = h->p.step_kernel;
    if (h->tma_ok && want != DBM_KERNEL_GENERIC) {
        const CUtensorMap *tm = &h->tmap[cur], *ti = &h->tmap_in[cur];
        if (h->tma_staged) return launch_staged(h, cur, fin, fout, st);
        switch (acc_mode(h->p)) {
        case 0: return launch_tma<0>(h, tm, ti, fin, fout, st);
        case 1: return launch_tma<1>(h, tm, ti, fin, fout, st);
        case 2: return launch_tma<2>(h, tm, ti, fin, fout, st);
        default: return launch_tma<3>(h, tm, ti, fin, fout, st);
        }
    }
    if (uses_acc(h->p)) return DBM_ERR_INVALID;  // the options exist in the TMA-staged kernel only
    if (want != DBM_KERNEL_AUTO && want != DBM_KERNEL_GENERIC) return DBM_ERR_INVALID;
    if (h->p.precision == DBM_BF16DEV) return launch_step_bf16(h, cur, st);
    if (h->p.precision == DBM_FP64) return launch_step_f64(h, cur, st);
    if (h->p.precision == DBM_FP32) return launch_generic(h, fin, fout, st);
    return DBM_ERR_INVALID;
}

}  // namespace dbm
