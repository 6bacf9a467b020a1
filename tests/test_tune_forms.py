"""What turtle_autotune times, on the CPU: csrc/tune.cu compiled as C++ with the counting call and the CUDA events
replaced by a model of the time, per form.

By tiles (the default form) the only knob with an effect is bucket_windows; the forms with a filter have all five, and a
class tuned in one form is not a class of the other."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

BODY = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#include "host.h"

static std::vector<turtle_params> seen;
static double (*cost)(const turtle_params &);

extern "C" {
void turtle_params_default(turtle_params *p) {
    memset(p, 0, sizeof(*p));
    p->struct_size = sizeof(*p);
    p->filter_bits_per_window = 1.0f;
    p->pattern_bits = 4;
    p->n_patterns = 1024;
}
int turtle_count_device(turtle_ctx *, const uint8_t *, uint64_t, const uint64_t *, uint64_t, int, uint32_t,
                        const turtle_params *p, void *, turtle_device_result *) {
    seen.push_back(*p);
    return TURTLE_OK;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = (float)cost(seen.back());
    return cudaSuccess;
}
}

static int bad = 0;
static void want(bool ok, const char *what) {
    if (!ok) bad++, fprintf(stderr, "%s\n", what);
}
static turtle_params tune(int k, uint32_t min_count, const turtle_params *base, turtle_tune_report *rep) {
    turtle_params best;
    uint64_t off[2] = {0, 1 << 20};
    uint8_t b = 0;
    seen.clear();
    want(turtle_autotune((turtle_ctx *)8, &b, 1 << 20, off, 1, k, min_count, base, nullptr, &best, rep) == TURTLE_OK, "rc");
    return best;
}
static uint32_t widest() {
    uint32_t w = 0;
    for (auto &p : seen) w = p.bucket_windows > w ? p.bucket_windows : w;
    return w;
}
static bool only_windows(const turtle_params &a) {
    for (auto p : seen) {
        p.bucket_windows = a.bucket_windows;
        p.timing = a.timing;
        if (memcmp(&p, &a, sizeof(a))) return false;
    }
    return true;
}

int main() {
    turtle_params d, p;
    turtle_tune_report rep;
    turtle_params_default(&d);
    // by tiles: bucket_windows alone, within a bucket's room, its optimum found
    cost = [](const turtle_params &q) {
        const double w = q.bucket_windows ? q.bucket_windows : 6400;
        return 10 + fabs(w - 4800) / 400 - (q.sort_tile == 2) - (q.bucket_slots == 4096) - (q.pattern_bits == 3);
    };
    p = tune(31, 2, nullptr, &rep);
    want(only_windows(d) && widest() <= 8192, "tiles, 64-bit keys: other knobs tried");
    want(p.bucket_windows == 4800 && rep.cached == 0 && rep.best_ms < rep.default_ms, "tiles, 64-bit keys: optimum");
    cost = [](const turtle_params &q) { return 10 + fabs((q.bucket_windows ? q.bucket_windows : 3200) - 2400.) / 400; };
    p = tune(55, 2, nullptr, &rep);
    want(only_windows(d) && widest() <= 8192 && p.bucket_windows == 2400, "tiles, 128-bit keys");
    // nothing to gain: the default stays, as 0
    cost = [](const turtle_params &q) { return q.bucket_windows ? 10.0 : 9.9; };
    turtle_tune_cache_clear();
    p = tune(31, 1, nullptr, &rep);
    want(p.bucket_windows == 0, "tiles: the default stays");
    // a form with a filter: all five knobs, a class of its own, and its knobs don't reach the form by tiles
    cost = [](const turtle_params &q) {
        return 20.0 - (q.sort_tile == 2) - (q.bucket_slots == 4096) - (q.pattern_bits == 3) - (q.bucket_windows == 32768);
    };
    turtle_tune_cache_clear();
    turtle_params f = d;
    f.probe_order = 1;
    p = tune(31, 2, &f, &rep);
    want(p.sort_tile == 2 && p.bucket_slots == 4096 && p.pattern_bits == 3 && p.bucket_windows == 32768, "filter: five knobs");
    p = tune(31, 2, &d, &rep);
    want(rep.cached == 0 && p.bucket_windows != 32768 && p.sort_tile == 0, "tiles: not the filter form's class");
    d.sort_tile = 3;  // a cached class gives the caller's other settings back as they were
    p = tune(31, 2, &d, &rep);
    want(rep.cached == 1 && p.sort_tile == 3, "tiles: cached");
    f.recount_windows = 1;
    f.probe_order = 0;
    tune(31, 1, &f, &rep);
    want(widest() <= 8192, "min_count 1 is counted by tiles whatever these say");
    printf("%d\n", bad);
}
"""


def test_each_form_is_tuned_by_its_own_knobs(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    csrc = os.path.join(ROOT, "paper_1305_1861_gb300", "csrc")
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(BODY)
    subprocess.run(["g++", "-std=c++17", "-O1", "-x", "c++", os.path.join(csrc, "tune.cu"), str(src), "-I", csrc, "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], check=True, capture_output=True, text=True)
    assert r.stdout.split() == ["0"], r.stderr
