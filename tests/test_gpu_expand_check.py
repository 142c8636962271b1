"""The depth-ordered binning's check of its own counts (needs a GB300).  No scene makes the counts
and the expansion disagree, so a small program linked with the library's objects calls the two
launchers with counts that do: k_expand must flag them, and the sort that gathers the records must
not read past the records, whatever the slots that were never written hold."""
import os
import subprocess

import pytest

from paper_1606_04427_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "splotch_internal.cuh"
#include <cstdio>
#include <vector>
using namespace spl;

template <typename T> static T *put(const std::vector<T> &h) {
    T *d = nullptr;
    cudaMalloc(&d, sizeof(T) * h.size());
    cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice);
    return d;
}
template <typename T> static std::vector<T> get(const T *d, size_t n) {
    std::vector<T> h(n);
    cudaMemcpy(h.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost);
    return h;
}

int main() {
    ViewParams v{};
    v.W = v.H = 32, v.T = 8, v.ntx = v.nty = 4, v.n_tiles = 16, v.hd = 0.70710677f * 8.0f;
    v.fastdiv = 1, v.tmagic = (uint32_t)((1ull << 32) / 8 + 1);
    ViewParams *views = put(std::vector<ViewParams>{v});
    // one tile, four tiles, all sixteen (expanded by the whole warp), none
    const int n = 4;
    float4 *prec = put(std::vector<float4>{{12, 12, 1, 0}, {16, 16, 2, 0}, {16, 16, 12, 0}, {-90, 0, 1, 0}});
    uint32_t *key = put(std::vector<uint32_t>{0, 1, 2, 3}), *pid = put(std::vector<uint32_t>{0, 1, 2, 3});
    float4 *srec = put(std::vector<float4>(n));
    uint32_t *cnt = put(std::vector<uint32_t>(n + 1));
    void *tmp = put(std::vector<char>(scan_temp_bytes(n + 1) + sort_temp_bytes(64)));
    launch_sorted_counts(views, prec, key, pid, n, 3u, srec, cnt, scan_arrivals(n + 1, tmp), 0);
    exclusive_scan_u32(cnt, n + 1, tmp, 0);
    const std::vector<uint32_t> off = get(cnt, n + 1);
    const int64_t P = off[n];
    printf("pairs %lld\n", (long long)P);
    auto expand = [&](const char *what, int from, int by, int64_t pairs) {
        std::vector<uint32_t> o = off;
        for (int k = from; k <= n; ++k) o[k] += by;  // particle from - 1 counted `by` tiles too many
        uint32_t *po = put(o), *tk = put(std::vector<uint32_t>(64, 77u)), *tv = put(std::vector<uint32_t>(64, 77u));
        int *status = put(std::vector<int>(4, 0));
        launch_expand(views, srec, po, (const uint32_t *)tmp, n, pairs, tk, tv, status, 0);
        const std::vector<uint32_t> k = get(tk, 64), t = get(tv, 64);
        bool past = false;
        for (int64_t j = pairs; j < 64; ++j) past |= k[j] != 77u || t[j] != 77u;
        printf("%s %d %d\n", what, get(status, 4)[kStatOverflow], (int)past);
    };
    expand("as-counted", 0, 0, P);
    for (int k = 1; k <= 4; ++k) expand("one-more", k, 1, P + 1);
    for (int k = 2; k <= 3; ++k) expand("one-fewer", k, -1, P - 1);
    expand("total-short", 0, 0, P + 1);
    expand("total-long", 0, 0, P - 1);
    // the gather of three records by places that include unwritten ones
    for (int m : {5, 1}) {
        std::vector<uint32_t> vals = {4000000000u, 1, 0, 3, 2};
        vals.resize(m);
        uint32_t *k0 = put(std::vector<uint32_t>(m, 5u)), *k1 = put(std::vector<uint32_t>(m)), *v0 = put(vals),
                 *v1 = put(std::vector<uint32_t>(m));
        float4 *out = put(std::vector<float4>(m));
        float4 *pay = put(std::vector<float4>{{10, 0, 0, 0}, {11, 0, 0, 0}, {12, 0, 0, 0}});
        radix_sort_gather(k0, k1, v0, v1, m, 0, 8, tmp, pay, 3, out, 0);
        printf("gather");
        for (float4 f : get(out, m)) printf(" %d", (int)f.x);
        printf("\n");
    }
    printf("%s\n", cudaGetErrorString(cudaDeviceSynchronize()));
    return 0;
}
"""


def test_expansion_flags_counts_that_disagree(tmp_path):
    build.build()
    objs = [os.path.join(build.OUT_DIR, s.replace(".cu", ".o")) for s in build.SOURCES if s != "splotch_api.cu"]
    src, exe = tmp_path / "expand.cu", tmp_path / "expand"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc()] + build.flags() + [str(src)] + objs + ["-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    assert out[0] == "pairs 21"
    assert out[1] == "as-counted 0 0"
    assert out[2:6] == ["one-more 1 0"] * 4
    assert out[6:8] == ["one-fewer 1 0"] * 2
    assert out[8:10] == ["total-short 1 0", "total-long 1 0"]
    assert out[10:12] == ["gather 12 11 10 12 12", "gather 12"]
    assert out[12] == "no error"
