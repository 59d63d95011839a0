"""The batch's counted compaction against the host for both widths of its tiles: sizes around
one tile, a word more or less, and around the line between the two, sparse and dense, and
more selected than there are slots."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fgs_internal.cuh"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace fgs;
#define OK(x) do { if ((x) != cudaSuccess) { std::printf("cuda error, line %d\n", __LINE__); return 1; } } while (0)
int main()
{
    const uint32_t sizes[] = {1, 31, 255, 1023, 1024, 1025, 40000, 1u << 22, (1u << 25) - 1, 1u << 25, (1u << 25) + 1,
                              (1u << 25) + 1025, (1u << 25) + 4097};
    const uint32_t max_words = (1u << 25) + 4097, max_cap = 20u << 20;
    uint32_t *d_bits, *d_sel, *d_cnt;
    FrameState* st;
    OK(cudaMalloc(&d_bits, 4ull * max_words));
    OK(cudaMalloc(&d_sel, 4ull * max_cap));
    OK(cudaMalloc(&d_cnt, 4ull * (max_words / 1024 + 1)));
    OK(cudaMalloc(&st, sizeof(FrameState)));
    uint64_t seed = 12345;
    auto next = [&] { return (uint32_t)((seed = seed * 6364136223846793005ull + 1442695040888963407ull) >> 32); };
    for (uint32_t n : sizes)
        for (int dense = 0; dense < 2; ++dense)
            for (int full = 0; full < 2; ++full) {
                std::vector<uint32_t> bits(n), want, cnt(batch_sel_tiles(n));
                for (uint32_t w = 0; w < n; ++w) {
                    bits[w] = dense ? (n > 1000000 ? next() & next() & next() & next() & next() & next() : next()) : next() % 997 == 0 ? next() : 0;
                    cnt[w / kBatchSelTileWords] += (uint32_t)__builtin_popcount(bits[w]);
                    for (int b = 0; b < 32; ++b)
                        if (bits[w] >> b & 1) want.push_back(32 * w + b);
                }
                if (want.size() > max_cap) return 2;
                const uint32_t cap = full ? (uint32_t)want.size() / 2 : max_cap, m = std::min((uint32_t)want.size(), cap);
                OK(cudaMemcpy(d_bits, bits.data(), 4ull * n, cudaMemcpyHostToDevice));
                OK(cudaMemcpy(d_cnt, cnt.data(), 4ull * cnt.size(), cudaMemcpyHostToDevice));
                OK(cudaMemset(d_sel, 0xFF, 4ull * max_cap));
                OK(cudaMemset(st, 0, sizeof(FrameState)));
                launch_compact_counted_batch(d_bits, n, d_sel, cap, d_cnt, st, 0);
                OK(cudaGetLastError());
                FrameState h;
                std::vector<uint32_t> got(max_cap);
                OK(cudaMemcpy(&h, st, sizeof h, cudaMemcpyDeviceToHost));
                OK(cudaMemcpy(got.data(), d_sel, 4ull * max_cap, cudaMemcpyDeviceToHost));
                const bool over = want.size() > cap;
                bool good = h.M == m && h.status == (over ? kErrCapacity : 0) && std::equal(want.begin(), want.begin() + m, got.begin());
                for (size_t i = m; i < got.size(); ++i) good = good && got[i] == 0xFFFFFFFFu;
                if (!good) std::printf("n %u dense %d full %d: M %u of %zu, status %d\n", n, dense, full, h.M, want.size(), h.status);
            }
    std::printf("done\n");
}
"""


def test_both_widths(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_23891_gb300 import build
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    (tmp_path / "c.cu").write_text(SOURCE)
    exe = str(tmp_path / "c")
    subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, str(tmp_path / "c.cu"), os.path.join(build.CSRC, "filter.cu"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout == "done\n", out.stdout
