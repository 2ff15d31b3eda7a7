"""CPU checks of the host rules that choose a launch (csrc/biot_args.h), compiled here
with the host compiler and evaluated over sizes and storage forms.

pair_takes_level is the one statement of which levels packed strips take: the launch of
a single instance instantiates and checks it, and the plan of a batch asks it, so a
batch never plans a packed sweep that its launch refuses.  pair_rows, pair_strip_ctas
and pair_frame_ctas: the strips and the frame's tiles cover every cell once.
"""
import itertools
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_11382_gb300", "csrc")


def evaluate(tmp_path, lines):
    """The ints that the C++ expressions print, one row per line."""
    from paper_2409_11382_gb300 import build as B
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    src = tmp_path / "rules.cpp"
    src.write_text('#include <stdio.h>\n#include "biot_args.h"\nusing namespace biot;\nint main()\n{\n' +
                   "\n".join(lines) + "\nreturn 0;\n}\n")
    exe = tmp_path / "rules"
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [[int(v) for v in line.split()] for line in out.splitlines()]


SIZES = [2, 6, 8, 10, 60, 62, 63, 64, 65, 66, 68, 124, 128, 250, 252, 256, 4094, 4096]


def test_packed_strips_take_the_levels_their_kernels_can_run(tmp_path):
    forms = list(itertools.product((0, 1), repeat=4))
    body = ["for (int fine = 0; fine < 2; fine++) for (int lo = 0; lo < 2; lo++) for (int gh = 0; gh < 2; gh++)",
            "for (int dev = 0; dev < 2; dev++) {",
            f"const int n[] = {{{', '.join(map(str, SIZES))}}};",
            'for (int nx : n) for (int ny : n) printf("%d ", (int)pair_takes_level(fine, lo, gh, dev, nx, ny));',
            'printf("\\n"); }']
    rows = evaluate(tmp_path, body)
    assert len(rows) == len(forms)
    for (fine, lo, gh, dev), row in zip(forms, rows):
        for (nx, ny), got in zip(itertools.product(SIZES, SIZES), row):
            # 16-byte copies of four FP32 cells, row pairs of the restriction, one 64-column
            # strip, rows above and below the frame; kernels exist without ghost moments and
            # deviation store, with low parts on the finest level alone
            can = nx % 4 == 0 and ny % 2 == 0 and nx >= 64 and ny >= 8 and not gh and not dev and lo == fine
            assert bool(got) == can, (fine, lo, gh, dev, nx, ny)


def test_plan_and_launch_ask_the_same_rule():
    def body(name, start):
        text = open(os.path.join(CSRC, name)).read()
        i = text.index(start)
        return text[i:text.index("\n}\n", i)]
    assert "pair_takes_level(" in body("biot_capi.cu", "bool level_takes_pair(const biot_ctx *h, int l, int v)\n{")
    assert "level_takes_pair(" in body("biot_capi.cu", "int op_variant(const biot_ctx *h, const PlanOp &o)\n{")
    assert "pair_takes_level(" in body("sweep_pair.cuh", "bool pair_takes(const SweepArgs<float, TC> &a)\n{")
    assert "pair_takes_level(" in body("sweep_mom.cuh", "cudaError_t launch_rows(")
    for name in ("biot_capi.cu", "sweep_pair.cuh", "sweep_mom.cuh"):  # and none restates it
        assert not re.search(r"nx % 4 == 0", open(os.path.join(CSRC, name)).read()), name


@pytest.mark.parametrize("slots", [4, 1824])
def test_strips_and_frame_cover_the_level_once(tmp_path, slots):
    sizes = [(64, 8), (64, 10), (68, 1000), (124, 66), (128, 256), (256, 256), (640, 520), (4096, 4096), (8192, 8)]
    body = [f"{{ const int nx = {nx}, ny = {ny}, ty = pair_rows(pair_strips_x(nx), ny - 4, {slots});\n"
            'printf("%d %d %d %d\\n", ty, pair_strips_x(nx), pair_strip_ctas(nx, ny, ty), pair_frame_ctas(nx, ny)); }'
            for nx, ny in sizes]
    rows = evaluate(tmp_path, body + ['printf("%d %d %d\\n", PAIR_WARPS, PAIR_COLS, PAIR_FX);'])
    warps, cols, fx = rows[-1]
    for (nx, ny), (ty, nsx, strips, frame) in zip(sizes, rows):
        assert ty >= 4 and ty % 2 == 0
        # columns 2 .. nx-3 in runs of `cols`, rows 2 .. ny-3 in runs of ty, one warp each
        assert (nsx - 1) * cols < nx - 4 <= nsx * cols
        blocks = -(-(ny - 4) // ty)
        assert strips == -(-nsx * blocks // warps)
        # two rows at the top and bottom, two columns at the sides, tiles of fx cells along them
        assert frame == 2 * -(-nx // fx) + 2 * -(-ny // fx)


def test_launch_code_keeps_no_plain_statics():
    """Instances are created and stepped from several threads (a server's worker among
    them), and a process may use several devices: what launch code remembers from its
    first launch is atomic and per device (DeviceCache), never a plain static."""
    plain = []
    for name in sorted(os.listdir(CSRC)):
        for i, line in enumerate(open(os.path.join(CSRC, name)), 1):
            if re.match(r"\s+static (?!const|constexpr|inline|DeviceCache|std::atomic)[\w:<>]+ \*?\w+( = [^;(]*)?;", line):
                plain.append(f"{name}:{i}: {line.strip()}")
    assert not plain, plain


def test_device_cache_is_one_number_per_device_from_many_threads(tmp_path):
    src = tmp_path / "cache.cpp"
    src.write_text(r"""
#include "biot_args.h"
#include <stdio.h>
#include <thread>
#include <vector>
static thread_local int current = 0;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
int main()
{
    static biot::DeviceCache c, failing;
    std::atomic<int> wrong{0}, calls{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 16; i++)
        t.emplace_back([&, i] {
            for (int k = 0; k < 20000; k++) {
                current = (i + k) % (biot::DeviceCache::DEVICES + 2);  // two beyond the table
                if (c.get([&](int dev) { calls++; return 100 + dev; }) != 100 + current) wrong++;
            }
        });
    for (auto &x : t) x.join();
    current = 3;
    const int f0 = failing.get([](int) { return 0; }), f1 = failing.get([](int) { return 7; });  // a failure is tried again
    printf("%d %d %d %d\n", wrong.load(), calls.load() >= biot::DeviceCache::DEVICES, f0, f1);
    return 0;
}
""")
    from paper_2409_11382_gb300 import build as B
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    exe = tmp_path / "cache"
    # under the thread sanitizer: a race in the cache ends the program with an error.  The
    # CUDA calls that the header's other functions name are never made here
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-pthread", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", str(exe),
           "-Wl,--unresolved-symbols=ignore-all"]

    def run(extra):
        if subprocess.run(cmd + extra, capture_output=True).returncode:
            return None
        return subprocess.run([str(exe)], capture_output=True, text=True)
    out = run(["-fsanitize=thread"])
    if out is None or "unexpected memory mapping" in out.stderr:  # no sanitizer on this host
        out = run([])
    assert out is not None and out.returncode == 0, out and out.stderr[-2000:]
    assert out.stdout.split() == ["0", "1", "0", "7"]


def test_packed_strips_take_the_tuned_height(tmp_path):
    """biot_autotune's height is the launch's, made even and at least four rows; without
    one the rule's.  The launch and the candidates of the tuner are the packed form's."""
    tuned = [0, -1, 1, 2, 3, 4, 5, 17, 64, 96, 158]
    got = evaluate(tmp_path, [f'printf("%d %d\\n", pair_height({t}, 69, 4092, 1824), pair_rows(69, 4092, 1824));'
                              for t in tuned])
    for t, (height, rule) in zip(tuned, got):
        assert height == (rule if t <= 0 else max(4, t + t % 2)), t
    pair = open(os.path.join(CSRC, "sweep_pair.cuh")).read()
    assert "pair_height(a.rows," in pair
    capi = open(os.path.join(CSRC, "biot_capi.cu")).read()
    tuner = capi[capi.index('extern "C" int biot_autotune(biot_handle h, int *rows_out'):]
    assert "level_takes_pair(" in tuner and "pair_rows_for(" in tuner
