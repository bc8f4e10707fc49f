"""The L-BFGS bookkeeping of the row solvers, whatever the order in which the
lanes of its warp run.

lbfgs_gram_update (solver_impl.cuh) is one warp's work on the row's scalars in
shared memory.  Between two __syncwarp() the lanes may run in any order, so no
lane may read there what another one writes.  This test compiles the function's
source for the host (no GPU), runs its 32 lanes as coroutines that change over
only at __syncwarp(), in ascending, descending and shuffled order, and asks for
the same state bit for bit, over rows with more pairs than the memory holds,
refused pairs and early stops."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_13524_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>
#include <ucontext.h>
struct int4 { int x, y, z, w; };
struct float4 { float x, y, z, w; };
static float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
using std::isfinite;
#define __device__
#define __forceinline__ inline
#define __align__(n) alignas(n)
static void __syncwarp();
constexpr int kMaxMem = 6, kMaxLanczos = 16;
@SOURCE@

// 32 lanes as coroutines; __syncwarp() hands over to the next lane in `order`
static ucontext_t main_ctx, ctx[32];
static std::vector<char> stacks[32];
static int current;
static bool finished[32];
static void __syncwarp() { swapcontext(&ctx[current], &main_ctx); }
struct Call { Gram *G; int m, it, iters; double tol; } call;
static void lane_main()
{
    const int lane = current;
    lbfgs_gram_update(*call.G, lane, call.m, call.it, call.iters, call.tol);
    finished[lane] = true;
}
static void warp(const std::vector<int> &order)
{
    for (int l = 0; l < 32; l++) {
        stacks[l].resize(64 << 10);
        getcontext(&ctx[l]);
        ctx[l].uc_stack.ss_sp = stacks[l].data();
        ctx[l].uc_stack.ss_size = stacks[l].size();
        ctx[l].uc_link = &main_ctx;
        makecontext(&ctx[l], lane_main, 0);
        finished[l] = false;
    }
    for (bool live = true; live;) {
        live = false;
        for (int l : order) {
            if (finished[l]) continue;
            current = l;
            swapcontext(&main_ctx, &ctx[l]);
            live = live || !finished[l];
        }
    }
}
int main()
{
    std::mt19937 rng(1);
    std::uniform_real_distribution<float> u(-1.f, 1.f);
    std::vector<std::vector<int>> orders(5, std::vector<int>(32));
    for (auto &o : orders)
        for (int l = 0; l < 32; l++) o[l] = l;
    std::reverse(orders[1].begin(), orders[1].end());
    for (int k = 2; k < 5; k++) std::shuffle(orders[k].begin(), orders[k].end(), rng);
    for (int m = 1; m <= kMaxMem; m++)
        for (int row = 0; row < 20; row++) {
            std::vector<Gram> G(orders.size());
            for (Gram &g : G) {
                std::memset(&g, 0, sizeof g);
                for (int i = 0; i < kGramPitch; i++) g.slot[i] = i;
                g.f = 100.f;
                g.gamma = 1.f;
            }
            const int iters = 3 * m + 4;
            for (int it = 0; it < iters; it++) {
                const int np = G[0].np;
                float red[kParts];
                for (float &x : red) x = 0.1f * u(rng);
                for (int i = 0; i <= np; i++) red[4 * i + 1] = 0.2f * u(rng);
                red[4 * np] = rng() % 5 ? 1.f + 0.2f * u(rng) : -1.f;  // one pair in five is refused
                red[4 * np + 1] = 2.f + u(rng);
                red[kIdxSS] = 1.f;
                red[kIdxGG] = 50.f;  // large: the direction stays one of descent
                red[kIdxF] = 90.f - it;
                for (size_t k = 0; k < G.size(); k++) {
                    std::memcpy(G[k].red, red, sizeof red);
                    call = {&G[k], m, it, iters, row % 2 ? 1e-9 : 0.0};
                    warp(orders[k]);
                    if (std::memcmp(&G[k], &G[0], sizeof(Gram))) {
                        std::printf("m %d, row %d, iteration %d: order %d differs\n", m, row, it, (int)k);
                        return 1;
                    }
                }
                bool seen[kSlots] = {};
                for (int i = 0; i <= m; i++) {
                    const int s = G[0].slot[i];
                    if (s < 0 || s > m || seen[s]) {
                        std::printf("m %d, row %d, iteration %d: slot %d twice or out of range\n", m, row, it, s);
                        return 1;
                    }
                    seen[s] = true;
                }
            }
        }
    std::printf("ok\n");
    return 0;
}
"""


def _source():
    with open(os.path.join(CSRC, "solver_impl.cuh")) as f:
        text = f.read()
    state = text[text.index("enum { ROW_MAXITER"):text.index("// Global minimiser of phi")]
    start = text.index("static __device__ void lbfgs_gram_update")
    return state + text[start:text.index("\n}\n", start) + 3]


def test_lane_order_does_not_matter(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "warp.cpp", tmp_path / "warp"
    src.write_text(PROGRAM.replace("@SOURCE@", _source()))
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-Wno-unknown-pragmas", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.stdout.strip() == "ok", out.stdout + out.stderr
