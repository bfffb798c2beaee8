"""The launchers hand a level and its parameters to kernels as objects of the
compute type's class (as_compute, csrc/qnsch_dev.cuh).  It copies the bits: the
copy equals its source byte for byte and does not change with it, and host code
that reads one class's object through a reference to the other does not build."""
import ctypes
import subprocess

from paper_1703_06606_gb300 import build

COPY = """
#include "qnsch_dev.cuh"
template <typename T, template <typename> class S>
static int same() {
  S<T> x;
  unsigned char* b = reinterpret_cast<unsigned char*>(&x);
  for (size_t k = 0; k < sizeof x; ++k) b[k] = (unsigned char)(k * 37 + 11);
  const auto y = qn::as_compute<qn::Fused<T>>(x);
  int bad = std::memcmp(&x, &y, sizeof x) != 0;
  for (size_t k = 0; k < sizeof x; ++k) b[k] = 0;
  const unsigned char* c = reinterpret_cast<const unsigned char*>(&y);
  for (size_t k = 0; k < sizeof x; ++k) bad |= c[k] != (unsigned char)(k * 37 + 11);
  return bad;
}
extern "C" int check() {
  return same<double, qn::Lv>() + 2 * same<float, qn::Lv>() + 4 * same<double, qn::Prm>() +
         8 * same<float, qn::Prm>();
}
"""
PUN = """
#include "qnsch_dev.cuh"
template <typename R, template <typename> class S, typename T>
static const S<R>& pun(const S<T>& x) {
  return reinterpret_cast<const S<R>&>(x);
}
extern "C" double first(const qn::Prm<double>& x) { return pun<qn::rf64>(x).ia.v; }
"""


def compile_host(text, tmp_path):
    src, out = tmp_path / "t.cu", tmp_path / "t.so"
    src.write_text(text)
    r = subprocess.run([build.nvcc()] + build.ARCH + build.HOST +
                       ["-O3", "-std=c++17", "-I", build.CSRC, "-shared", "-o", str(out), str(src)],
                       capture_output=True, text=True)
    return r, out


def test_the_copy_has_the_bits(tmp_path):
    r, out = compile_host(COPY, tmp_path)
    assert r.returncode == 0, r.stderr
    assert ctypes.CDLL(str(out)).check() == 0


def test_reading_another_class_does_not_build(tmp_path):
    r, _ = compile_host(PUN, tmp_path)
    assert r.returncode != 0 and "strict-aliasing" in r.stderr
