"""The bisection of dev::brick_run against a walk over every candidate sample,
on the host: the same function, compiled for the CPU, must give the run that the
ownership test itself gives sample by sample, for rays parallel and nearly
parallel to faces, axis-aligned directions, grazing rays, eyes inside and on
boundaries, steps from a hundredth of a voxel to many voxels, and bricks on and
off the volume's faces."""
import os
import subprocess

from paper_2501_01628_gb300 import build

HARNESS = r'''
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include "vr_device.cuh"
using namespace vr;
struct P { float dt, inv_dt, nmax, N[3]; };

// a ray as ray_setup leaves it
static void make_ray(const P &p, const float o[3], const float d[3], dev::Ray &r)
{
    float t0 = 0.f, t1 = 3.0e38f, dmin = 3.0e38f;
    bool hit = true;
    for (int i = 0; i < 3; ++i) {
        r.ov[i] = o[i] * p.nmax;
        r.dv[i] = d[i] * p.nmax;
        r.inv[i] = 0.f;
        if (r.dv[i] == 0.f) {
            if (r.ov[i] < 0.f || r.ov[i] > p.N[i]) hit = false;
            continue;
        }
        r.inv[i] = 1.0f / r.dv[i];
        const float ta = (0.f - r.ov[i]) * r.inv[i], tb = (p.N[i] - r.ov[i]) * r.inv[i];
        t0 = std::fmax(t0, std::fmin(ta, tb));
        t1 = std::fmin(t1, std::fmax(ta, tb));
        dmin = std::fmin(dmin, std::fabs(r.dv[i]));
    }
    r.t_in = t0;
    r.t_out = t1;
    r.hit = hit && t0 < t1;
    r.margin = 2 + static_cast<int>(std::fmin(2.0e4f, 1.0e-6f * p.nmax / (dmin * p.dt)));
}

// the run by trying every candidate; false where the brick owns no sample
static bool walk(const P &p, const BrickLaunch &B, const dev::Ray &r, int &ka, int &kb)
{
    if (!r.hit) return false;
    float b0 = 0.f, b1 = 3.0e38f;
    for (int i = 0; i < 3; ++i) {
        if (r.dv[i] == 0.f) {
            if (r.ov[i] < B.lo[i] || r.ov[i] > B.hi[i]) return false;
            continue;
        }
        const float ta = (static_cast<float>(B.lo[i]) - r.ov[i]) * r.inv[i];
        const float tb = (static_cast<float>(B.hi[i]) - r.ov[i]) * r.inv[i];
        b0 = std::fmax(b0, std::fmin(ta, tb));
        b1 = std::fmin(b1, std::fmax(ta, tb));
    }
    if (!(b0 <= b1)) return false;
    ka = std::max(0, static_cast<int>(std::floor((b0 - r.t_in) * p.inv_dt - 0.5f)) - r.margin);
    kb = static_cast<int>(std::ceil((std::fmin(b1, r.t_out) - r.t_in) * p.inv_dt - 0.5f)) + r.margin;
    auto owned = [&](int k) {
        const float t = std::fmaf(static_cast<float>(k) + 0.5f, p.dt, r.t_in);
        bool in = t < r.t_out;
        for (int i = 0; i < 3; ++i) {
            const float q = std::fmaf(t, r.dv[i], r.ov[i]);
            in = in && q >= B.own_lo[i] && q < B.own_hi[i];
        }
        return in;
    };
    while (ka <= kb && !owned(ka)) ++ka;
    while (kb > ka && !owned(kb)) --kb;
    return ka <= kb;
}

int main()
{
    std::mt19937 rng(7);
    std::uniform_real_distribution<float> u(0.f, 1.f);
    auto pick = [&](std::initializer_list<float> v) { return v.begin()[rng() % v.size()]; };
    long runs = 0, empty = 0, wide = 0, bad = 0;
    for (int it = 0; it < 400000; ++it) {
        int N[3], lo[3], hi[3];
        for (int i = 0; i < 3; ++i) {
            N[i] = 1 + rng() % 200;
            lo[i] = rng() % 2 ? 0 : static_cast<int>(rng() % N[i]);
            hi[i] = rng() % 2 ? N[i] : lo[i] + 1 + static_cast<int>(rng() % (N[i] - lo[i]));
        }
        P p;
        p.nmax = static_cast<float>(std::max(N[0], std::max(N[1], N[2])));
        BrickLaunch B{};
        for (int i = 0; i < 3; ++i) {
            p.N[i] = static_cast<float>(N[i]);
            B.lo[i] = lo[i];
            B.hi[i] = hi[i];
            B.own_lo[i] = lo[i] == 0 ? -INFINITY : static_cast<float>(lo[i]);
            B.own_hi[i] = hi[i] == N[i] ? INFINITY : static_cast<float>(hi[i]);
        }
        const double dt = pick({0.5f, 0.5f, 0.37f, 1.0f, 0.05f, 0.01f, 4.3f, 50.f}) / p.nmax;
        p.dt = static_cast<float>(dt);
        p.inv_dt = static_cast<float>(1.0 / dt);
        float o[3], d[3], l = 0.f;
        for (int i = 0; i < 3; ++i) {
            // through the box from anywhere, with components of every smallness
            d[i] = (u(rng) * 2.f - 1.f) * pick({1.f, 1.f, 1.f, 1e-2f, 1e-4f, 1e-6f, 1e-7f, 1e-9f, 0.f});
            l += d[i] * d[i];
        }
        if (l == 0.f) continue;
        const float s = pick({0.f, 0.f, 0.5f, 2.f, 2.f, 2.f});
        for (int i = 0; i < 3; ++i) {
            d[i] /= std::sqrt(l);
            float target = p.N[i] / p.nmax * (u(rng) * 1.1f - 0.05f);
            if (rng() % 4 == 0) target = (rng() % 2 ? lo[i] : hi[i]) / p.nmax;  // on a face
            o[i] = target - s * d[i];
        }
        dev::Ray r;
        make_ray(p, o, d, r);
        dev::OwnedRun run;
        dev::brick_run(p, B, r, run);
        int ka = 0, kb = -1;
        const bool any = walk(p, B, r, ka, kb);
        const bool same = any ? run.ka == ka && run.kb == kb : run.ka > run.kb;
        if (!same && bad++ < 5) std::printf("it %d: [%d, %d] against [%d, %d] (any %d)\n", it, run.ka, run.kb, ka, kb, any);
        runs += any;
        empty += !any;
        wide += any && r.margin > 100;
    }
    std::printf("runs %ld empty %ld wide margins %ld bad %ld\n", runs, empty, wide, bad);
    return bad || runs < 50000 || empty < 20000 || wide < 5000;
}
'''


def test_search_equals_walk(tmp_path):
    src = tmp_path / "owned_run_check.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "owned_run_check"
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, "-o", str(exe), str(src)],
                   check=True, cwd=os.path.dirname(build.CSRC))
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
