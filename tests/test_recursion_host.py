"""The helicity-shared recursion, compiled for the host, against the
per-helicity program of the same process (no GPU).

The kernels of the larger processes build the colour flows by a colour-ordered
recursion whose currents are shared between helicities
(generator/recursion.py, csrc/mg_recursion.cuh).  Run here with one thread on
the host, stage by stage, it must give, for every helicity, every colour flow
of the diagram-by-diagram program (up to one common phase) and its colour form.

Tolerance: both sum the same Feynman diagrams in the same gauge; their flows
differ by the rounding of up to ~1e3 terms, each at most ~1e2 times the
largest flow of its helicity: 1e3 * 1e2 * 1.1e-16 = 1e-11 of that flow.
"""
import subprocess

import numpy as np
import pytest

from paper_2303_18244_gb300.generator import emit, recursion
from paper_2303_18244_gb300.inputs import process_momenta
from test_generated_code_host import CSRC, _couplings

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __restrict__
template <typename T> inline T __ldg(const T* p) { return *p; }
#include "TAG.cuh"
#include "TAG_rec.cuh"
using namespace mg;
using P = TAG_rec;
using ST = rec::Store<double, P::N, P::NVEC<double>>;
int main() {
  double kp[8];
  for (double& x : kp)
    if (scanf("%lf", &x) != 1) return 1;
  int nevt;
  if (scanf("%d", &nevt) != 1) return 1;
  void* mem = aligned_alloc(128, (ST::bytes + 255) / 128 * 128);
  const ST st(mem);
  for (int e = 0; e < nevt; e++) {
    double p[P::NPAR * 4];
    for (double& x : p)
      if (scanf("%lf", &x) != 1) return 1;
    std::vector<double> slab(TAG::NSLOT);
    TAG::prepare<double, double>(p, kp, slab.data(), 1);
    for (int m = 0; m < ST::NSUB; m++) rec::setup_momenta<P, double>(st, p, m);
    for (int c = 0; c < 2 * ST::NSUB; c++) rec::setup_coef<P, double, double>(st, p, kp, c);
    for (int l = 0; l < P::N + 2; l++) rec::setup_leg<P, double>(st, p, kp, l);
    CURRENTS
    for (int hg = 0; hg < (1 << P::N); hg++)
      for (int s = 0; s < 2; s++) {
        static cx<double> a[2][P::NCOL];
        FLOWS
        for (int b = 0; b < 2; b++) {
          const int h = P::helicity(hg, s, b);
          static cx<double> jamp[P::NCOL];
          TAG::amplitudes<double>(slab.data(), 1, h, kp, jamp, 1);
          // the recursion leaves out the common factor i
          double worst = 0.0, big = 0.0;
          for (int k = 0; k < P::NCOL; k++) {
            const cx<double> j = jamp[LEX(k)];
            worst = std::fmax(worst, std::hypot(-a[b][k].im - j.re, a[b][k].re - j.im));
            big = std::fmax(big, std::hypot(j.re, j.im));
          }
          const double v = P::colour_form<double>(a[b]);
          printf("%d %.17g %.17g %.17g\n", h, big > 0 ? worst / big : worst, v,
                 TAG::colour_quadratic<double>(jamp, 1));
        }
      }
  }
  return 0;
}
"""


def _run(proc, sqrts, nevt, workdir):
    tag, n = emit.PROCESSES[proc]
    (workdir / f"{tag}.cuh").write_text(emit.emit(proc, "f64")[1])
    (workdir / f"{tag}_rec.cuh").write_text(recursion.emit_recursion(n, tag))
    src = PROGRAM.replace("CURRENTS", recursion.HOST_CURRENTS[n > 4]).replace("FLOWS", recursion.HOST_FLOWS[n > 4])
    src = src.replace("LEX(k)", "P::lex_flow(k)" if n > 4 else "k")
    (workdir / "main.cpp").write_text(src.replace("TAG", tag))
    exe = workdir / "main"
    subprocess.run(["g++", "-O0", "-std=c++17", f"-I{workdir}", f"-I{CSRC}", "-o", str(exe),
                    str(workdir / "main.cpp")], check=True)
    p = process_momenta(proc, sqrts, nevt, 57)
    lines = [" ".join(repr(float(x)) for x in _couplings(proc)), str(nevt)]
    lines += [" ".join(repr(float(x)) for x in ev.ravel()) for ev in p]
    out = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True).stdout
    return np.array([[float(x) for x in ln.split()] for ln in out.splitlines()]).reshape(nevt, 1 << (n + 2), 4)


@pytest.mark.parametrize("proc,sqrts,nevt", [("g g > t t~", 1000.0, 20), ("g g > t t~ g", 1200.0, 10),
                                             ("g g > t t~ g g", 1500.0, 6), ("g g > t t~ g g g", 2000.0, 1)],
                         ids=["ggtt", "ggttg", "ggttgg", "ggttggg"])
def test_flows_of_every_helicity(proc, sqrts, nevt, tmp_path):
    r = _run(proc, sqrts, nevt, tmp_path)
    nhel = r.shape[1]
    for e in range(nevt):
        assert sorted(r[e, :, 0].astype(int)) == list(range(nhel))  # every helicity once
        assert np.max(r[e, :, 1]) <= 1e-11
        tot = r[e, :, 3].sum()
        assert np.max(np.abs(r[e, :, 2] - r[e, :, 3])) <= 1e-11 * tot


THREAD_PROGRAM = PROGRAM[:PROGRAM.index('#include "TAG.cuh"')] + r"""
#include "TAG.cuh"
REC
using namespace mg;
int main() {
  double kp[8];
  for (double& x : kp)
    if (scanf("%lf", &x) != 1) return 1;
  int nevt;
  if (scanf("%d", &nevt) != 1) return 1;
  for (int e = 0; e < nevt; e++) {
    double p[TAG::NPAR * 4];
    for (double& x : p)
      if (scanf("%lf", &x) != 1) return 1;
    unsigned good;
    if (scanf("%u", &good) != 1) return 1;
    double slab[TAG::NSLOT], want = 0.0;
    TAG::prepare<double, double>(p, kp, slab, 1);
    for (int h = 0; h < TAG::NHEL; h++)
      if (good >> h & 1u) {
        cx<double> jamp[TAG::NCOL];
        TAG::amplitudes<double>(slab, 1, h, kp, jamp, 1);
        want += TAG::colour_quadratic<double>(jamp, 1);
      }
    printf("%.17g %.17g\n", THREAD::thread_sum<double, double, double>(p, kp, good), want);
  }
  return 0;
}
"""


@pytest.mark.parametrize("proc,sqrts,rec", [("g g > t t~", 1000.0, True), ("u u~ > t t~ g", 1200.0, False)],
                         ids=["ggtt", "uuttg"])
def test_thread_sum_over_helicity_lists(proc, sqrts, rec, tmp_path):
    """One thread's sum over all helicities, for the full list, single
    helicities and random lists, against the per-helicity program summed over
    the same list (1e-12: the sum of a list can be a small part of its
    helicities' currents, each within 1e-14 or so of the program's)."""
    tag, n = emit.PROCESSES[proc]
    (tmp_path / f"{tag}.cuh").write_text(emit.emit(proc, "f64")[1])
    src = THREAD_PROGRAM.replace("REC", f'#include "{tag}_rec.cuh"' if rec else "")
    if rec:
        (tmp_path / f"{tag}_rec.cuh").write_text(recursion.emit_recursion(n, tag))
    (tmp_path / "main.cpp").write_text(src.replace("THREAD", f"{tag}_rec" if rec else tag).replace("TAG", tag))
    exe = tmp_path / "main"
    subprocess.run(["g++", "-O0", "-std=c++17", f"-I{tmp_path}", f"-I{CSRC}", "-o", str(exe), str(tmp_path / "main.cpp")],
                   check=True)
    nhel = 1 << len(proc.replace(">", " ").split())
    rng = np.random.default_rng(3)
    lists = [(1 << nhel) - 1] + [1 << h for h in range(nhel)] + [int(rng.integers(1, 1 << nhel)) for _ in range(10)]
    p = process_momenta(proc, sqrts, len(lists), 58)
    lines = [" ".join(repr(float(x)) for x in _couplings(proc)), str(len(lists))]
    lines += [" ".join(repr(float(x)) for x in ev.ravel()) + f" {m}" for ev, m in zip(p, lists)]
    out = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True).stdout
    r = np.array([[float(x) for x in ln.split()] for ln in out.splitlines()])
    assert r.shape == (len(lists), 2) and np.all(r[0] > 0)
    zero = r[:, 1] == 0.0  # equal u and u~ helicities: exactly zero on both sides
    assert np.all(r[zero, 0] == 0.0)
    assert np.max(np.abs(r[~zero, 0] / r[~zero, 1] - 1)) <= 1e-12
