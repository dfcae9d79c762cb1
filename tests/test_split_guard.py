"""The y,z stage's split of a row item between two halves of the thread groups branches on a
group's line around the transforms' warp barriers, so every warp's lines must lie on one
side.  The guard is evaluated at compile time over the real line order, which permutes
groups in blocks of 16: with TPL = 8, lines 0..3 and 4..7 share the first warp although
4 is a multiple of the four groups of a warp.
"""
import subprocess

from paper_1505_05341_gb300 import build

PROGRAM = """
#include "fft.cuh"
#include "spectra.cuh"
using namespace ys;
static_assert(!warps_on_one_side<8>(64, 4) && !warps_on_one_side<4>(64, 8) && !warps_on_one_side<2>(128, 8));
static_assert(warps_on_one_side<8>(32, 16) && warps_on_one_side<4>(64, 32) && warps_on_one_side<2>(128, 32));
static_assert(warps_on_one_side<32>(8, 4) && warps_on_one_side<64>(8, 3) && !warps_on_one_side<16>(16, 5));
template <int N, int ELL> constexpr bool sound() {
  using Y = YZ<N, ELL>;
  return !Y::SPLIT || warps_on_one_side<Y::TPL>(Y::GROUPS, Y::R);
}
static_assert(sound<16, 6>() && sound<32, 4>() && sound<32, 6>() && sound<64, 6>() && sound<96, 6>() && sound<128, 6>());
static_assert(sound<192, 6>() && sound<256, 6>() && sound<384, 6>() && sound<512, 4>() && sound<512, 6>() && sound<1024, 4>());
static_assert(YZ<32, 4>::SPLIT && YZ<128, 6>::SPLIT && YZ<256, 6>::SPLIT);
"""


def test_guard(tmp_path):
    src = tmp_path / "guard.cu"
    src.write_text(PROGRAM)
    r = subprocess.run([build._nvcc(), *build.FLAGS, *build.ARCH, "-I", build.CSRC, "-I", build.HERE + "/../include", "-c",
                        "-o", str(tmp_path / "guard.out"), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
