"""The host's rules that choose a kernel, a tile or a schedule, on the CPU."""
import ctypes
import os
import subprocess

from paper_2402_08725_gb300 import build


def _run_cpp(tmp_path, body, head='#include "kernels.cuh"\n'):
    """Integers printed by the statements `body`, compiled against the library's internal headers."""
    src, exe = tmp_path / "rule.cu", str(tmp_path / "rule")
    src.write_text("#include <cstdio>\n" + head + "int main() {\n" + body + "\n}\n")
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", exe], check=True)
    return [int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]


def test_an_epoch_without_a_second_pairs_its_phases(tmp_path):
    """Transforms of the kernel spectra: one per phase of two epochs, half as many for a single one."""
    calls = "".join(f'  printf("%d\\n", sr::fft_kappa_items({E}, {f}));\n' for E in (1, 2, 3, 8) for f in (1, 2, 3))
    assert _run_cpp(tmp_path, calls) == [1, 2, 5, 1, 4, 9, 2, 6, 14, 4, 16, 36]


def _rule(name):
    """A host function of the library that no C header declares."""
    from paper_2402_08725_gb300 import _native
    return getattr(ctypes.CDLL(_native.load()._name), name)


def _ints(v):
    return (ctypes.c_int * len(v))(*v)


def test_tile_height_is_the_tables():
    """A field that leaves SMs idle alone takes short tiles; the same field in a batch that fills them does not
    pay their halo."""
    rows = _rule("_ZN2sr9tile_rowsEPKiS1_iii")
    for n, want in ((1, 16), (4, 16), (8, 32), (16, 32), (32, 64)):
        assert rows(_ints([24] * n), _ints([64] * n), n, 152, 0) == want
    assert rows(_ints([300]), _ints([64]), 1, 152, 0) == 32
    assert rows(_ints([]), _ints([]), 0, 152, 0) == 16


def test_the_form_autotuner_times_the_tiles_of_full_batches():
    """Its verdict is kept by shape, for any number of epochs: the first field's must not enter it."""
    rows = _rule("_ZN2sr9tile_rowsEPKiS1_iii")
    assert {rows(_ints([E]), _ints([64]), 1, 152, 1) for E in (1, 4, 16)} == {64}


def test_clusters_only_where_they_do_not_queue():
    """Starlet clusters: grids up to 256 pixels, in tables whose clusters do not wait long for one another."""
    bits, cluster = _rule("_ZN2sr22starlet_comb_rows_bitsEPKiS1_ii"), 128

    def has(F, J):
        return bool(bits(_ints(F), _ints(J), len(F), 152) & cluster)

    assert has([64], [4]) and has([128] * 12, [4] * 12) and has([256], [4]) and has([420, 128], [5, 4])
    assert has([64, 96, 128] * 8, [4, 5, 6] * 8)
    assert not has([64] * 16, [4] * 16) and not has([128] * 32, [6] * 32) and not has([64, 96] * 19, [4, 6] * 19)
    assert not has([420], [5]) and not has([600, 300], [5, 5])


def test_shift_gradient_threads_follow_the_grid(tmp_path):
    """About 16 pixels a thread, whole warps, 128 to 1024 threads."""
    got = _run_cpp(tmp_path, "".join(f'  printf("%d\\n", sr::hshift_threads({F}));\n' for F in (5, 64, 90, 128, 1536)))
    assert got == [128, 256, 512, 1024, 1024]


def test_each_device_is_set_up_once(tmp_path):
    """A second device gets its own set-up, a failed one is repeated, and threads together run it once."""
    head = """#include <atomic>
#include <thread>
#include <vector>
#include "once.cuh"
namespace sr { sr_status cuda_fail(cudaError_t, const char *) { return SR_ERR_CUDA; } }
"""
    body = """
  sr::OncePerDevice once;
  std::atomic<int> n{0};
  auto ok = [&] { ++n; return SR_OK; };
  auto bad = [&] { ++n; return SR_ERR_CUDA; };
  printf("%d ", (int)once.run_on(0, bad));
  once.run_on(0, ok); once.run_on(0, ok); printf("%d ", n.load());   // failed, then done once
  once.run_on(1, ok); once.run_on(1, ok); printf("%d ", n.load());   // another device
  once.run_on(63, ok); once.run_on(63, ok); once.run_on(64, ok); once.run_on(64, ok); printf("%d ", n.load());
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k) t.emplace_back([&] { once.run_on(2, ok); });
  for (auto &x : t) x.join();
  printf("%d", n.load());
"""
    assert _run_cpp(tmp_path, body, head) == [4, 2, 3, 6, 7]


def test_the_kernels_of_every_file_are_set_up_per_device():
    """No kernel attribute or constant table is set behind a once-per-process flag."""
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as fh:
            text = fh.read()
        assert "once_flag" not in text and "static std::atomic<bool>" not in text, name


def test_items_are_priced_by_the_groups_they_run_in():
    """Epochs per item: where nine phases leave no room for two pairs the pairs of an item share no passes."""
    epochs, group = _rule("_ZN2sr16fft_chunk_epochsEPKNS_8FftShapeEiii"), _rule("_ZN2sr14fft_pair_groupEiiiii")
    limit = 229500

    def item(L, M, f, E):
        return epochs(_ints([L, M, f, E]), 1, 152, limit)

    assert group(112, 1, 2, 0, limit) == 2 and group(112, 1, 3, 0, limit) == 1 and group(112, 1, 2, 1, limit) == 1
    assert group(32, 1, 2, 0, limit) == 4 and group(32, 2, 2, 0, limit) == 1
    assert item(112, 1, 2, 300) == 4 and item(112, 1, 3, 300) == 2 and item(32, 1, 2, 1000) == 8
    assert epochs(_ints([]), 0, 152, limit) == 2
