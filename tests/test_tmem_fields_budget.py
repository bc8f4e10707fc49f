"""Host-side check of the tensor-memory columns that the row solver allocates
once the row's fields wait there beside the L-BFGS pairs, with one CTA per row
and over a cluster (solver_row.cuh).

A CTA that finds too few free columns waits for another one to give its own
back.  So the columns of all CTAs that share an SM have to fit in 512, and a
cluster's CTA, whose neighbour may be waiting for it, may share its SM with
none of its kind."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_13524_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "solver_row.cuh"
using namespace tmr;
static void line(const char *kind, int N, int J, int JB, int nloc, size_t smem)
{
    const RowShape s = row_shape(N, JB, nloc);
    for (int m = 1; m <= kMaxMem; m++)
        for (int k = 0; k <= kMaxLanczos; k++) {
            const int klz = s.klz(k > 0, k);
            std::printf("%s %d %d %d %d %d %d %d %d %d %d %d %d %zu\n", kind, N, J, JB, m, k, s.threads, s.ept, klz,
                        s.quarter_warps(), s.cols(m, klz, true), s.cols(m, klz, false), (int)row_fields_fit(s, m, klz), smem);
        }
}
int main()
{
    for (int N : {512, 1024, 2048, 4096})
        for (int J = 1; J <= kMaxMasks; J++) {
            if (N <= 2048 && row_variant_fits(N, J))
                line("row", N, J, J, N, N == 512 ? row_smem<512>(J, 5) : N == 1024 ? row_smem<1024>(J, 5) : row_smem<2048>(J, 5));
            if (const int JB = rowc_masks(N, J))
                line("cluster", N, J, JB, (N + J / JB - 1) / (J / JB), N == 2048 ? rowc_smem<2048>(J) : rowc_smem<4096>(J));
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    nvcc = next((c for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc")
                 if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fields")
    (d / "fields.cu").write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                        os.path.join(ROOT, "include"), "-I", CSRC, str(d / "fields.cu"), "-o", str(d / "fields")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(d / "fields")], capture_output=True, text=True, check=True).stdout
    return [(f[0], *map(int, f[1:])) for f in (x.split() for x in out.splitlines())]


def test_the_cluster_shapes(table):
    assert {(N, J, JB) for kind, N, J, JB, *_ in table if kind == "cluster"} == {
        (4096, 4, 2), (4096, 6, 2), (4096, 8, 2), (2048, 6, 3), (2048, 8, 4)}


def test_the_columns_hold_what_a_cta_keeps(table):
    for kind, N, J, JB, m, k, threads, ept, klz, qw, cols, bare, fit, _ in table:
        nloc = -(-N // (J // JB))
        assert threads == JB * N // 16 <= 512 and threads % 32 == 0
        assert ept * threads >= nloc > (ept - 1) * threads
        for c, z in ((cols, 32), (bare, 0)):  # 16 complex values a thread
            assert c >= 32 and c & (c - 1) == 0
            assert c >= qw * (4 * ept * (m + 1) + z) and (not klz or c >= qw * 2 * ept * klz)
        assert bare <= 512 and (not fit or cols <= 512)  # with the fields only where they fit


def test_the_fields_take_no_resident_cta_away(table):
    for kind, N, J, JB, m, k, threads, ept, klz, qw, cols, bare, fit, _ in table:
        by_registers = 512 // threads
        resident = min(by_registers, 512 // bare)
        assert fit == (cols <= 512 and 512 // cols >= resident)


def test_a_cluster_cta_is_alone_on_its_sm(table):
    # 228 KB of shared memory an SM; the launch asks for at least 116 KB, the kernel for what it needs
    for kind, N, J, JB, m, k, *_, fit, smem in table:
        if kind == "cluster" and fit:
            assert smem <= 227 * 1024 and 2 * max(smem, 116 * 1024) > 228 * 1024
