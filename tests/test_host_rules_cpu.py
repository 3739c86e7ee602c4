"""Host-side rules of the launchers that no launch on one device can reach, compiled from the headers into a small program (no device call is made)."""
import os
import subprocess

import pytest

from paper_2203_16487_b200 import build

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <tuple>
#include "vocab_rows.cuh"

// a map that carries its base address: what encoding leaves in it is this test's own
static CUresult fake_encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void* base, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                            CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    memset(m, 0, sizeof *m);
    memcpy(m, &base, sizeof base);
    return CUDA_SUCCESS;
}
static bool is_of(const CUtensorMap& m, const void* base) { return !memcmp(&m, &base, sizeof base); }

// A launch's two maps, asked for while the cache is at its limit: both are what was asked for.
static int maps_of_one_launch() {
    sd::TmaEncoder enc;
    enc.encode = fake_encode;
    int wrong = 0;
    for (long long i = 1; i < 20000; ++i) {
        CUtensorMap a, w;
        const void *pa = (const void*)(i << 20), *pw = (const void*)((i << 20) + 4096);
        wrong += !enc.get(a, pa, i, 512, 512, 128) || !enc.get(w, pw, 512, 512, 512, 64) || !is_of(a, pa) || !is_of(w, pw);
        CUtensorMap again;                               // ... from the cache, or encoded once more
        wrong += !enc.get(again, pa, i, 512, 512, 128) || !is_of(again, pa);
        if (enc.cache.size() > 5000) ++wrong;
    }
    return wrong;
}

// The few-rows vocabulary kernel: CTA r of the grid stores row r, so there are as many tiles as rows wherever it is used; on 148 SMs every count up to 32 is.
static int rows_without_a_cta() {
    int wrong = 0;
    sd::TmaEncoder enc;
    enc.ready = true;
    for (enc.n_sm = 1; enc.n_sm <= 200; ++enc.n_sm)
        for (int N = 128; N <= 50000; N += 97)
            for (int rows = 1; rows <= 33; ++rows)
                wrong += sd::vr_supported(enc, N, 512, rows) && (N + sd::VR_BN - 1) / sd::VR_BN < rows;
    enc.n_sm = 148;
    for (int N = 18000; N <= 34000; ++N)
        for (int rows = 1; rows <= 33; ++rows) wrong += sd::vr_supported(enc, N, 512, rows) != (N > 148 * 128 && N <= 148 * 224 && rows <= 32);
    return wrong;
}

int main() {
    printf("rows_without_a_cta %d\n", rows_without_a_cta());
    printf("maps_of_one_launch %d\n", maps_of_one_launch());
    return 0;
}
"""


@pytest.fixture(scope="module")
def wrong(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_rules")
    src, exe = d / "rules.cu", d / "rules"
    src.write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-I", build.CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    env = dict(os.environ, MALLOC_PERTURB_="165", GLIBC_TUNABLES="glibc.malloc.tcache_count=0")        # what is freed does not keep its contents
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True, timeout=60, env=env).stdout
    return dict((name, int(n)) for name, n in (line.split() for line in out.splitlines()))


def test_the_maps_of_a_launch_survive_the_eviction_between_them(wrong):
    assert wrong["maps_of_one_launch"] == 0


def test_every_row_of_the_few_rows_vocabulary_kernel_has_a_cta(wrong):
    assert wrong["rows_without_a_cta"] == 0


@pytest.mark.parametrize("kg,kw,message", [
    (4, 32, None),
    (2, 64, "8-column tiles"),                           # would leave half of the output's columns zero
    (4, 16, "no second pass"),                           # would leave out the keys beyond its one block
])
def test_key_groups_share_probabilities_in_the_forms_the_kernel_handles(kg, kw, message, tmp_path):
    src = tmp_path / "k.cu"
    src.write_text('#include "attention.cuh"\n'
                   f"template __global__ void sd::k_attn<false, 1, {kg}, {kw}, 3, true>(sd::AttnTcArgs, sd::QueryArgs, sd::OutArgs);\n")
    r = subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I" + build.CSRC, "-cubin",
                        "-o", str(tmp_path / "k.out"), str(src)], capture_output=True, text=True)
    assert (r.returncode == 0) == (message is None) and (message or "") in r.stderr, r.stderr
