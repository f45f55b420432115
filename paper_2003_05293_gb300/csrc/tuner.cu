// Autotuner of the FP32 iteration kernels' tile shapes (compressed
// iterations: threads per block and pixels per thread; full passes: threads
// per block).  Key: (largest P rounded up to 128, work-weighted spot
// count rounded up to a power of two, batch size rounded up to a power of
// two, subset fraction c as the nearest power of two: a compressed launch on
// the CUDA cores costs c times a full one, on the tensor cores about as much
// as a full one, so the winner changes with c; and whether the pupil is round
// and the beam Gaussian, since a round pupil has fewer pixels and dearer draws:
// the paper's optics take 769 us a solve with the direct-phasor shape that is
// best on a square of their size and 634 with their own).  Each candidate runs a
// synthetic batch of that key's size (three compressed iterations in a row, or
// one full iteration and the final pass; as a graph, like a user's run); the
// fastest compressed-iteration shape and the fastest full-pass shape win, with
// a handicap of the tensor cores.  Results live in the plan and, when the
// plan names a cache file, in a small JSON file.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>

#include "runtime.h"

namespace cswgs {

cswgs_status batch_build_with(cswgs_plan_s *p, std::vector<HoloSpec> specs, TileShape shape,
                              std::unique_ptr<Fp32Batch> *out);

static int pow2_ceil(int x)
{
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

struct TuneKey {
    int P, N, B;
    int cexp;   // c = 2^-cexp (0 .. 16)
    bool round, beam;   // most of the work under a round pupil, a Gaussian beam
};

// The subset fraction of a batch, weighted by each hologram's compressed
// work (pixels x spots x compressed iterations); 1 when none has any.
static double batch_c(const std::vector<HoloSpec> &specs)
{
    double wsum = 0.0, cw = 0.0;
    for (auto &s : specs) {
        const int F = std::min(s.n_full, s.iterations);
        const double M = (double)s.P * s.P, D = s.D > 0 ? (double)s.D : M;
        const double w = M * s.N * (double)(s.iterations - F), c = (double)s.Mp / D;
        wsum += w;
        cw += w * c;
    }
    return wsum > 0.0 ? cw / wsum : 1.0;
}

static TuneKey key_of(const std::vector<HoloSpec> &specs)
{
    int P = 0;
    double wsum = 0.0, nw = 0.0, round = 0.0, beam = 0.0;
    for (auto &s : specs) {
        P = std::max(P, s.P);
        double w = (double)s.P * s.P * s.N;
        wsum += w;
        nw += w * s.N;
        round += s.aperture == CSWGS_APERTURE_ROUND ? w : 0.0;
        beam += s.waist > 0.0 ? w : 0.0;
    }
    int N = wsum > 0 ? (int)std::lround(nw / wsum) : 1;
    TuneKey k;
    k.P = ((P + 127) / 128) * 128;
    k.N = std::max(16, pow2_ceil(N));
    k.B = pow2_ceil((int)specs.size());
    const double c = batch_c(specs);
    k.cexp = std::min(16, std::max(0, (int)std::lround(-std::log2(std::max(c, 1e-9)))));
    k.round = 2.0 * round > wsum;
    k.beam = 2.0 * beam > wsum;
    return k;
}

// The key's name: "P1152_N64_B1_c3", then "_R" (round), "_G" (Gaussian), "_H"
// (half precision); `pupil` false leaves the pupil's letters out.
static std::string tune_key(const TuneKey &k, bool fp16, bool pupil = true)
{
    char buf[64];
    snprintf(buf, sizeof buf, "P%d_N%d_B%d_c%d%s%s%s", k.P, k.N, k.B, k.cexp, pupil && k.round ? "_R" : "",
             pupil && k.beam ? "_G" : "", fp16 ? "_H" : "");
    return buf;
}

// Candidates: compressed-iteration kernel (threads, pixels per thread, the
// masked tensor-core pass, or the subset-only gather kernel) and full-pass
// kernel (threads, or a tensor-core kernel); the two kinds run as separate launches, so each is tuned on its
// own launches.
static const int kSubCandidates[][2] = {{128, 2}, {128, 4}, {128, 8}, {256, 2},  {256, 4},
                                        {256, 8}, {512, 1}, {512, 2}, {512, 4}, {kSubsetTc, 1},
                                        {kSubsetGather, 1}};
static const int kFullCandidates[] = {128, 256, 512, kFullTcWs};

// Compressed iterations of a timed run: in a row, since a chain's launches
// overlap and the next mask is drawn beside them (a single iteration launched
// kernel by kernel timed the launches of small work, not the work, and the
// choice changed from run to run: one optics' solves took 680 or 870 us).
constexpr int kTuneSub = 3;

// The tensor cores' products keep 16 bits of their operands and drop what falls
// below FP32's last bit, the CUDA cores' kernels work in FP32: the pick is part
// of what a caller gets for a size.  So it keeps to the lines that the timings
// drew when the tensor-core launches started up serially and summed a hologram's
// partials on one SM, rather than move with each gain of those launches: a
// tensor-core launch's time counts with what it cost more then, net of the other
// kernels' gains (medians over 432 sizes, P = 128 to 1152, N = 16 to 512, c = 1 to
// 1/32, batches of 1 to 64; ms, by the key's N and B).  Without it 51 of these
// sizes take the tensor cores for compressed iterations and 163 for a final pass
// that did not before, and a whole solve of P = 64 came out 1.1e-5 from exact
// instead of 1.5e-6; with it 3 and 8 do, and 13 and 8 the other way round (of those
// timings' own picks, 5 % differed from one run to the next).
static double tc_sub_extra(const TuneKey &k) { return 1e-3 * (4.0 + k.N / 40.0 + 1.5 * std::log2(k.B)); }
static double tc_full_extra(const TuneKey &k) { return 1e-3 * (4.5 + k.N / 50.0); }
static double tc_final_extra(const TuneKey &k) { return 1e-3 * (26.0 + k.N / 25.0 + 3.0 * std::log2(k.B)); }

// A synthetic batch of the key's size: kTuneSub compressed iterations, or a full
// iteration and the final pass.
static cswgs_status synthetic(cswgs_plan_s *p, const TuneKey &k, double c, bool full, std::vector<HoloSpec> *out)
{
    HoloSpec pupil;
    pupil.P = std::min(k.P, 4096);
    cswgs_pupil pu{};
    pu.aperture = k.round ? CSWGS_APERTURE_ROUND : CSWGS_APERTURE_SQUARE;
    pu.beam_waist = k.beam ? 0.5 * pupil.P : 0.0;
    CSWGS_TRY(apply_pupil(p, pu, std::max(c, 2.0 / ((double)pupil.P * pupil.P)), &pupil));   // one pixel at least
    out->clear();
    for (int b = 0; b < k.B; ++b) {
        HoloSpec s = pupil;
        s.N = k.N;
        s.iterations = full ? 1 : kTuneSub;
        s.n_full = full ? 1 : 0;
        s.first_j = 1;
        s.final_pass = full ? 1 : 0;
        s.seed = 0x5EEDull + (uint64_t)b;
        s.xyz.resize(3 * (size_t)s.N);
        uint64_t x = 12345 + (uint64_t)b;
        for (auto &q : s.xyz) {
            x = x * 6364136223846793005ull + 1442695040888963407ull;
            q = ((double)(x >> 11) * 0x1.0p-53 - 0.5) * (s.P / 2.0);
        }
        out->push_back(std::move(s));
    }
    return CSWGS_OK;
}

// Device times (ms) of the synthetic schedule's parts: a compressed iteration,
// or a full iteration and the final pass, each the best of three runs after a
// warm-up; a candidate that takes half as long again as `best` (three times as
// long in the warm-up), by cost(t), is not run again.
template <class Cost>
static cswgs_status time_steps(cswgs_plan_s *p, const std::vector<HoloSpec> &specs, TileShape sh, bool full,
                               double best, Cost cost, double t[2])
{
    std::unique_ptr<Fp32Batch> b;
    CSWGS_TRY(batch_build_with(p, specs, sh, &b));
    b->joined_steps = full ? 1 : kTuneSub;
    b->test_hook = false;
    CSWGS_TRY(batch_upload_inputs(b.get(), p->stream));
    t[0] = t[1] = 1e30;
    for (int rep = 0; rep < 4; ++rep) {
        CSWGS_TRY(batch_enqueue(b.get(), p->stream));
        CSWGS_CUDA_TRY(cudaStreamSynchronize(p->stream));
        double r[2] = {0.0, 0.0};
        for (int i = 0; i < (full ? 2 : 1); ++i) {
            float ms = 0.f;
            CSWGS_CUDA_TRY(cudaEventElapsedTime(&ms, b->events[1 + i], b->events[full ? 2 + i : 1 + kTuneSub]));
            r[i] = full ? ms : ms / kTuneSub;
        }
        const bool slow = cost(r) > (rep == 0 ? 3.0 : 1.5) * best;   // a first run is a cold one
        if (rep == 0 && !slow) continue;
        for (int i = 0; i < 2; ++i) t[i] = std::min(t[i], r[i]);
        if (slow) break;
    }
    return CSWGS_OK;
}

static cswgs_status tune_for(cswgs_plan_s *p, const TuneKey &k, double c, double wsub, double wfull,
                             TileShape *best_shape, double *best_ms)
{
    const int fp16 = p->desc.precision == CSWGS_FP32_FP16SINCOS ? 1 : 0;
    TileShape best{256, 4, 256, fp16};
    double best_sub = 1e30, best_full = 1e30, ms_sub = 0.0, ms_full = 0.0, t[2];
    std::vector<HoloSpec> specs;
    CSWGS_TRY(synthetic(p, k, c, false, &specs));
    for (const auto &cand : kSubCandidates) {
        TileShape sh{cand[0], cand[1], best.full_threads, fp16};
        if (!shape_supported(sh)) continue;
        if (shape_max_grid(sh, kLaunchSubset, k.N, p->sm_count) <= 0) continue;
        const double extra = cand[0] == kSubsetTc ? tc_sub_extra(k) : 0.0;
        const auto cost = [&](const double *r) { return r[0] + extra; };
        CSWGS_TRY(time_steps(p, specs, sh, false, best_sub, cost, t));
        if (cost(t) < best_sub) {
            best_sub = cost(t);
            ms_sub = t[0];
            best.threads = cand[0];
            best.ppt = cand[1];
        }
    }
    CSWGS_TRY(synthetic(p, k, c, true, &specs));
    for (int ft : kFullCandidates) {
        TileShape sh{best.threads, best.ppt, ft, fp16};
        if (shape_max_grid(sh, kLaunchFull, k.N, p->sm_count) <= 0) continue;
        const double extra = is_full_tc(ft) ? wfull * tc_full_extra(k) + tc_final_extra(k) : 0.0;
        const auto cost = [&](const double *r) { return wfull * r[0] + r[1] + extra; };
        CSWGS_TRY(time_steps(p, specs, sh, true, best_full, cost, t));
        if (cost(t) < best_full) {
            best_full = cost(t);
            ms_full = wfull * t[0] + t[1];
            best.full_threads = ft;
        }
    }
    *best_shape = best;
    if (best_ms) *best_ms = wsub * ms_sub + ms_full;
    return CSWGS_OK;
}

TileShape tuned_shape(cswgs_plan_s *p, const std::vector<HoloSpec> &specs)
{
    const bool fp16 = p->desc.precision == CSWGS_FP32_FP16SINCOS;
    const TuneKey k = key_of(specs);
    const std::string key = tune_key(k, fp16);
    auto it = p->tune.find(key);
    if (it == p->tune.end() && p->tune_any_pupil) it = p->tune.find(tune_key(k, fp16, false));
    if (it != p->tune.end()) return it->second;
    // tune now, with the schedule's own mix of compressed and full iterations
    double wsub = 0.0, wfull = 0.0;
    for (auto &s : specs) {
        int F = std::min(s.n_full, s.iterations);
        wsub += s.iterations - F;
        wfull += F;
    }
    const double c = std::ldexp(1.0, -k.cexp);   // the key's c: one tuning per bucket
    if (!specs.empty()) {
        wsub /= specs.size();
        wfull /= specs.size();
    }
    TileShape sh{256, 4, 256, fp16 ? 1 : 0};
    double ms = 0.0;
    if (tune_for(p, k, c, wsub, wfull, &sh, &ms) == CSWGS_OK) {
        p->tune[key] = sh;
        tune_save(p);
    }
    return sh;
}

cswgs_status tune_single(cswgs_plan_s *p, int P, int N, double c, double *best_ms)
{
    HoloSpec s;
    s.P = P;
    s.N = N;
    s.Mp = std::max(1, (int)std::floor(c * (double)P * P));
    s.iterations = 30;
    s.n_full = 2;
    std::vector<HoloSpec> v{s};
    TuneKey k = key_of(v);
    TileShape sh;
    CSWGS_TRY(tune_for(p, k, c, 28.0, 2.0, &sh, best_ms));
    p->tune[tune_key(k, p->desc.precision == CSWGS_FP32_FP16SINCOS)] = sh;
    tune_save(p);
    return CSWGS_OK;
}

void tune_load(cswgs_plan_s *p)
{
    if (p->tune_path.empty()) return;
    std::ifstream f(p->tune_path);
    if (!f) return;
    std::stringstream ss;
    ss << f.rdbuf();
    std::string s = ss.str();
    // entries look like "P1152_N128_B64_c3": [256, 4, 128] or, with a strip
    // length for the tensor-core launches, [1, 1, 2, 6]
    size_t pos = 0;
    while ((pos = s.find('"', pos)) != std::string::npos) {
        size_t end = s.find('"', pos + 1);
        if (end == std::string::npos) break;
        std::string key = s.substr(pos + 1, end - pos - 1);
        pos = end + 1;
        if (key.empty() || key[0] != 'P') continue;
        const int fp16 = key.size() > 2 && key.compare(key.size() - 2, 2, "_H") == 0 ? 1 : 0;
        int t = 0, k = 0, f = 0, st = 0;
        const int got = sscanf(s.c_str() + pos, " : [ %d , %d , %d , %d ]", &t, &k, &f, &st);
        if (got < 3) continue;
        if (got < 4 || st < 0 || st > 4096) st = 0;
        if (shape_supported(TileShape{t, k, f, fp16, st})) p->tune[key] = TileShape{t, k, f, fp16, st};
    }
    // files before format 4 have no pupil in their keys: an entry holds for every pupil
    p->tune_any_pupil = !p->tune.empty() && s.find("\"cswgs-tune-4\"") == std::string::npos;
}

void tune_save(cswgs_plan_s *p)
{
    if (p->tune_path.empty()) return;
    std::string tmp = p->tune_path + ".tmp";
    FILE *f = fopen(tmp.c_str(), "w");
    if (!f) return;
    fprintf(f, "{\n  \"format\": \"cswgs-tune-%d\",\n  \"entries\": {", p->tune_any_pupil ? 3 : 4);
    bool first = true;
    for (auto &kv : p->tune) {
        fprintf(f, "%s\n    \"%s\": [%d, %d, %d, %d]", first ? "" : ",", kv.first.c_str(), kv.second.threads,
                kv.second.ppt, kv.second.full_threads, kv.second.strip);
        first = false;
    }
    fprintf(f, "\n  }\n}\n");
    fclose(f);
    rename(tmp.c_str(), p->tune_path.c_str());
}

}  // namespace cswgs
