// Host checks of the C interface's host code (celeste_api.cu) on a stand-in for the CUDA runtime,
// the launchers of the other files replaced by ones that record what they were asked for.
// Argument: which check.  Exit status 1 on a failure.
//   memory   The device memory of a problem: the Hessian pass's part records take the place of
//            the per-pixel E_s / Var_s, which its map passes are done with by then.
//   settled  A problem's counters and flags are filled when its creation returns: the fills are
//            on the default stream, which an evaluation on a non-blocking stream does not wait for.
//   autotune The map pass is timed as the paths that take the choice run it: at the multiply
//            covered pixels (the Hessian evaluation) and at every pixel without the maps (a fit's batches).
#include "fake_runtime.cuh"

#include "celeste_api.cu"

namespace cel {
cudaError_t launch_prep(const DevProblem&, const double*, int, cudaStream_t, bool, bool) { return cudaSuccess; }
static std::map<int, int> hess_passes, fit_passes, other_passes;   // by kernel code
cudaError_t launch_contrib(const DevProblem& P, int, cudaStream_t, bool multi_only) {
    ++(P.single && multi_only ? hess_passes : !P.single && !multi_only ? fit_passes : other_passes)[P.tune_contrib];
    return cudaSuccess;
}
cudaError_t launch_gather(const DevProblem&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_adjoint(const DevProblem&, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_hess_pixels(const DevProblem&, int, const double*, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finalize(const DevProblem&, const double*, int, int, double*, double*, double*, double*, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_items_stage(const DevProblem&, int, int, cudaStream_t, const double*, double*, double*, double*) {
    return cudaSuccess;
}
cudaError_t launch_catalog(int, const double*, double*, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_score(int, const double*, const double*, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fill_sky(const DevProblem&, double*, double*, cudaStream_t) { return cudaSuccess; }
void prime_persistent_grids() {}
cudaError_t prime_items_kernels() { return cudaSuccess; }
cudaError_t prime_hess_kernels() { return cudaSuccess; }
celeste_status fit_sources_impl(celeste_problem*, double*, const int32_t*, int32_t, const celeste_fit_options*, int32_t*,
                                int32_t*, double*, celeste_status (*)(celeste_problem*, const double*, int32_t, double*, double*),
                                const int32_t*) {
    return CELESTE_ERR_CUDA;
}
}  // namespace cel
extern "C" void celeste_fit_options_default(celeste_fit_options* o) { *o = celeste_fit_options{}; }

// five bands of side x side pixels; n sources, patches of w x w from a row-major grid of pitch
// (w: no overlaps)
static celeste_problem* create(int side, int n, int w, int pitch) {
    static std::vector<float> px;
    px.assign((size_t)side * side, 100.f);
    static const double psf[18] = {0.5, 0, 0, 2, 0, 2, 0.3, 0, 0, 4, 0, 4, 0.2, 0, 0, 9, 0, 9};
    std::vector<celeste_image> im(5);
    for (int b = 0; b < 5; ++b) {
        im[b] = celeste_image{};
        im[b].band = b;
        im[b].height = im[b].width = side;
        im[b].pixels = px.data();
        im[b].sky = 100;
        im[b].nmgy_per_count = 0.005;
        im[b].wcs[0] = im[b].wcs[3] = 1;
        im[b].n_psf = 3;
        im[b].psf = psf;
    }
    double mix[2][8][2], prior_r[4] = {0, 1, 0, 1}, prior_c[2][8][21] = {};
    for (auto& m : mix)
        for (int j = 0; j < 8; ++j) m[j][0] = 0.125, m[j][1] = 0.1 * (j + 1);
    for (auto& t : prior_c)
        for (auto& c : t) {
            c[0] = 0.125;
            for (int j = 0; j < 4; ++j) c[5 + 5 * j] = 1;
        }
    const celeste_model model{6, 8, &mix[0][0][0], &mix[1][0][0], 0.5, prior_r, 8, &prior_c[0][0][0]};
    std::vector<int32_t> off(n + 1), nbr(n + 1, 0);
    std::vector<celeste_patch> patch;
    const int row = (side - w) / pitch + 1;
    for (int s = 0; s < n; ++s) {
        off[s] = 5 * s;
        for (int b = 0; b < 5; ++b) patch.push_back({b, s % row * pitch, s / row * pitch, w, w});
    }
    off[n] = 5 * n;
    celeste_problem* pr = nullptr;
    const celeste_status st =
        celeste_problem_create(im.data(), 5, &model, n, off.data(), patch.data(), nbr.data(), nullptr, &pr);
    if (st != CELESTE_OK) printf("create: %d %s\n", st, celeste_last_error());
    return pr;
}

static int check_memory() {
    celeste_problem* pr = create(1024, 210, 31, 40);
    if (!pr) return 1;
    const DevProblem& P = pr->P;
    if (P.hchunk != 128) return printf("parts of %d pixels\n", P.hchunk), 1;
    const size_t held = fake::live_bytes;
    const size_t pixel = 4 + 16, sp = 16 + 16 + 1;   // counts and maps; E_s and Var_s, item records, flags
    const size_t patch = 8 * TBL_STRIDE + 4 * TBL_STRIDE + 4 * ZFULL_FLOATS + 16 * ZCHAIN + sizeof(PatchGeo) + sizeof(ZBuild) + 8;
    const size_t source = 8 * (2 * NP + 2 + HREC + 1 + NP + NP * NP) + 4 + 8;
    const size_t may = pixel * P.n_px + sp * P.n_sp + patch * P.n_patch + source * P.n_src + P.n_item * (sizeof(WorkItem) + 8 * NPART + 8) +
                       P.n_hitem * sizeof(HItem) + P.n_sitem * (sizeof(ZTask) + 128) + sizeof(ZTask) +
                       sizeof(ImgMeta) * P.n_img_rec + sizeof(ModelDev) + sizeof(ZCand) * P.n_zcand + P.n_tile * (sizeof(Tile) + 8) +
                       4 * (P.n_tile_list + P.n_tile_grid) + 8192;
    printf("%zu %zu\n", held, may);
    celeste_problem_destroy(pr);
    return held <= may && fake::live_bytes == 0 ? 0 : 1;
}

static int check_settled() {
    celeste_problem* pr = create(128, 4, 9, 20);
    if (!pr) return 1;
    const int n = fake::unsettled;
    if (n) printf("%d fills under way\n", n);
    celeste_problem_destroy(pr);
    return n != 0;
}

static int check_autotune() {
    celeste_problem* pr = create(128, 4, 9, 20);
    if (!pr) return 1;
    std::vector<double> theta((size_t)pr->P.n_src * NP, 0.5);
    const celeste_status st = celeste_autotune(pr, theta.data(), 3, nullptr, nullptr);
    bool ok = st == CELESTE_OK && cel::other_passes.empty() && cel::hess_passes.size() == 7 &&
              cel::hess_passes == cel::fit_passes;
    printf("status %d, codes: Hessian %zu, fit %zu, neither %zu\n", st, cel::hess_passes.size(), cel::fit_passes.size(),
           cel::other_passes.size());
    celeste_problem_destroy(pr);
    return ok ? 0 : 1;
}

int main(int argc, char** argv) {
    fake::no_real_device();
    const char* what = argc > 1 ? argv[1] : "";
    if (!strcmp(what, "memory")) return check_memory();
    if (!strcmp(what, "settled")) return check_settled();
    if (!strcmp(what, "autotune")) return check_autotune();
    printf("unknown check %s\n", what);
    return 1;
}
