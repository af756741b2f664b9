// Host check of the device memory that a fit takes (fit.cu) on a stand-in for the CUDA runtime:
// argument "fp64", "fp32" (with the FP64 polish) or "fp32only", then "colour" or "cyclades".
// Prints the bytes held when the first evaluation of the problem is due (every buffer is in place
// then) and what they may be: per pixel of the largest batch six values, per patch one table
// of the widest precision used, per part of the Hessian pass its record.
#include "fake_runtime.cuh"

#include "fit.cu"

namespace cel {
#define STUB { return cudaErrorNotSupported; }
cudaError_t launch_prep(const DevProblem&, const double*, int, cudaStream_t, bool, bool) STUB
cudaError_t launch_contrib(const DevProblem&, int, cudaStream_t, bool) STUB
cudaError_t launch_hess_pixels(const DevProblem&, int, const double*, double*, cudaStream_t) STUB
cudaError_t launch_finalize_hess(const DevProblem&, int, double*, double*, double*, cudaStream_t) STUB
void set_last_error(const char*) {}
}  // namespace cel

static size_t held = 0;
static celeste_status first_evaluation(celeste_problem*, const double*, int32_t, double*, double*) {
    held = fake::live_bytes;
    return CELESTE_ERR_TIMEOUT;   // (ends the fit)
}

int main(int argc, char** argv) {
    fake::no_real_device();
    if (argc < 3) return 1;
    const std::string prec = argv[1], sched = argv[2];
    // 4000 sources of five images each, no two patches overlapping: one colour, and large
    // enough for parts of 128 pixels; every third patch is of 31 x 31 pixels, the others 23 x 23
    const int n = 4000, n_img = 5;
    celeste_problem pr;
    pr.P.n_src = n;
    pr.P.n_patch = n * n_img;
    pr.imgs.resize(n_img);
    for (auto& im : pr.imgs) im.W = im.H = 4096, im.npsf = 3;
    size_t pixels = 0, parts = 0, items = 0;
    const int side[3] = {31, 23, 23}, chunk = 128;
    for (int s = 0; s < n; ++s) {
        pr.patch_off.push_back((int)pr.geo.size());
        pr.nbr_off.push_back(0);
        for (int i = 0; i < n_img; ++i) {
            cel::PatchGeo g{};
            g.img = i;
            g.w = g.h = side[pr.geo.size() % 3];
            g.src = s;
            g.sp_off = (int64_t)pixels;
            pr.geo.push_back(g);
            const int px = g.w * g.h;
            pixels += px;
            parts += (px + chunk - 1) / chunk;
            items += (px + cel::CHUNK - 1) / cel::CHUNK;
        }
    }
    pr.patch_off.push_back((int)pr.geo.size());
    pr.nbr_off.push_back(0);
    pr.P.n_sp = (int64_t)pixels;
    std::vector<double> theta((size_t)n * cel::NP, 0.5), d_theta(theta.size());
    pr.d_theta = d_theta.data();
    celeste_fit_options o;
    celeste_fit_options_default(&o);
    o.precision = prec == "fp64" ? CELESTE_FP64 : CELESTE_FP32_ACC64;
    o.refine_fp64 = prec == "fp32";
    o.schedule = sched == "colour" ? CELESTE_SCHED_COLOUR : CELESTE_SCHED_CYCLADES;
    o.sample_size = n;
    const celeste_status st = cel::fit_sources_impl(&pr, theta.data(), nullptr, 0, &o, nullptr, nullptr, nullptr, first_evaluation);
    const size_t patches = pr.geo.size(), table = prec == "fp32only" ? 3584 : 6656;
    const size_t may = 48 * pixels + patches * (table + sizeof(cel::PatchGeo)) + items * (sizeof(cel::WorkItem) + 8) +
                       parts * (8 * cel::HV + sizeof(cel::HItem)) +
                       n * (8 * (2 * cel::NP + 2 * cel::NT + 2 + cel::NP + cel::NP * cel::NP + cel::HREC) + 12 + sizeof(cel::TrState)) + 4096;
    printf("%zu %zu\n", held, may);
    return st == CELESTE_ERR_TIMEOUT && held > 0 && held <= may && fake::live_bytes == 0 ? 0 : 1;
}
