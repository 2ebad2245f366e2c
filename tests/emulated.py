"""The library's host functions and its generated kernels on the CPU: a program around
csrc/chem_host.cpp (the code generator and the layout rules), and the generated source compiled with
lane_emulator.h."""
import os
import re
import subprocess

import numpy as np

from tests.conftest import ROOT

HERE = os.path.dirname(os.path.abspath(__file__))


def host_program(tmp, main, name="host", flags=()):
    """An executable of `main` (C++ text) compiled together with chem_host.cpp."""
    from paper_2205_05681_gb300 import build as b
    b.build()
    src = os.path.join(str(tmp), name + ".cpp")
    with open(src, "w") as fh:
        fh.write('#include "%s"\n%s' % (os.path.join(b.CSRC, "chem_host.cpp"), main))
    exe = os.path.join(str(tmp), name)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", b.OUT_DIR,
                           "-I", os.path.join(b.CUDA, "include"), *flags, src, "-o", exe,
                           "-L", os.path.join(b.CUDA, "lib64"), "-Wl,-rpath," + os.path.join(b.CUDA, "lib64"),
                           "-lnvrtc", "-ldl", "-lpthread"])
    return exe


EMIT = r"""
int main(int, char** v) {
  MechData d;
  if (read_spec(v[1], &d)) { fprintf(stderr, "%s\n", g_last_error.c_str()); return 1; }
  fputs(emit_mechanism(d, atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5])).c_str(), stdout);
}
"""

# inline PTX -> the emulator's functions
PTX = [(r'asm volatile\("bar\.sync 1, %0;" ::"r"\((.*?)\) : "memory"\);', r"emu_bar(1, \1);"),
       (r'asm\("sub\.f16x2 %0, %1, %2;" : "=r"\((.*?)\) : "r"\((.*?)\), "r"\((.*?)\)\);', r"\1 = emu_hsub2(\2, \3);"),
       (r'asm\("mma\.sync\.aligned\.m16n8k16.*?;"\s*:.*?;', "emu_mma16(c, a0, a1, a2, a3, b0, b1);"),
       (r'asm\("mma\.sync\.aligned\.m16n8k8\..*?;"\s*:.*?;', "emu_mma8(c, a0, a1, b0);")]

DRIVER = r"""
double smem[1 << 16];
static std::vector<double> arr(size_t n) {
  std::vector<double> v(n);
  if (fread(v.data(), 8, n, stdin) != n) exit(4);
  return v;
}
static void put(const std::vector<double>& v) { fwrite(v.data(), 8, v.size(), stdout); }
int main(int, char** argv) {
  const int order = atoi(argv[1]);
  const long long n = atoll(argv[2]);
  std::fill(smem, smem + (1 << 16), __longlong_as_double(0x7ff8000000000000LL));
  std::vector<double> T = arr(n), P = arr(n), X = arr((size_t)NS * n);
  bool ok = true;
  %s
  fflush(stdout);
  return ok ? 0 : 5;
}
"""
# X: moles n[k][cell]
EVAL = r"""
  std::vector<double> f(NS * n), J(NS * NS * n), A = arr(NR);
  const double* lnA = atoi(argv[3]) ? A.data() : nullptr;
  ok = emu::run(TPB, order, [&] { chem_eval_source_k(n, T.data(), P.data(), X.data(), f.data(), n, lnA); });
  ok = ok && emu::run(TPB, order, [&] { chem_eval_jacobian_k(n, T.data(), P.data(), X.data(), J.data(), n, lnA); });
  put(f); put(J);
"""
# X: moles; then the weights v[k][cell]
VJP = r"""
  std::vector<double> v = arr((size_t)NS * n), gy(NS * n), gp(NR * n);
  ok = emu::run(TPB, order, [&] { chem_eval_vjp_k(n, T.data(), P.data(), X.data(), v.data(), gy.data(), gp.data(), n, nullptr); });
  put(gy); put(gp);
"""
# X: mass fractions Y[k][cell]; with argv[6] a cache of the W-method's factors
INTEGRATE = r"""
  std::vector<double> h(n), C(WC_STRIDE * n);
  std::vector<int> status(n, -1), att(n, -1);
  unsigned long long q = 0;
  ok = emu::run(TPB, order, [&] {
    chem_integrate_k(n, T.data(), P.data(), X.data(), n, atof(argv[3]), atof(argv[4]), atof(argv[5]), h.data(),
                     status.data(), att.data(), nullptr, 1000, 1e-20, 0.0, &q, nullptr, nullptr, nullptr, 0, 0,
                     nullptr, nullptr, 0, nullptr, 0, atoi(argv[6]) ? C.data() : nullptr); });
  put(T); put(X); put(C); put(h);
  put(std::vector<double>(status.begin(), status.end())); put(std::vector<double>(att.begin(), att.end()));
"""


class Emulated:
    """The generated kernels of one mechanism and launch configuration on the CPU."""

    def __init__(self, tmp, emit, spec, team, block, body, adjoint=False, tableau=0):
        src = subprocess.run([emit, spec, str(team), str(block), str(int(adjoint)), str(tableau)],
                             capture_output=True, text=True, check=True).stdout
        for a, b in PTX:
            src = re.sub(a, b, src, flags=re.S)
        src = re.sub(r"#ifndef FX_HOST.*?#endif", "", src, flags=re.S)
        assert "asm" not in src
        path = os.path.join(str(tmp), "k%d_%d_%d_%d.cpp" % (team, block, adjoint, tableau))
        with open(path, "w") as fh:
            fh.write('#include "%s"\n%s\n%s' % (os.path.join(HERE, "lane_emulator.h"), src, DRIVER % body))
        self.exe = path[:-4]
        subprocess.check_call(["g++", "-O1", "-std=gnu++17", "-w", "-ffp-contract=off", path, "-o", self.exe])
        self.team = team

    def _run(self, args, arrays):
        r = subprocess.run([self.exe] + [str(a) for a in args], capture_output=True, timeout=600,
                           input=b"".join(np.ascontiguousarray(a, dtype=np.float64).tobytes() for a in arrays))
        assert r.returncode == 0, "lanes stuck:\n" + r.stderr.decode()[-2000:]
        return np.frombuffer(r.stdout)

    def eval(self, T, P, n, nr, lnA=None, order=1):
        """f [cell, Ns] and J [cell, Ns, Ns]; n [cell, Ns - 1]"""
        c, ns = len(T), n.shape[1] + 1
        X = np.zeros((ns, c))
        X[:-1] = n.T
        o = self._run([order, c, int(lnA is not None)], [T, P, X, np.zeros(nr) if lnA is None else lnA])
        return o[:ns * c].reshape(ns, c).T, o[ns * c:].reshape(ns * ns, c).T.reshape(c, ns, ns)

    def vjp(self, T, P, n, v, order=1):
        """J^T v [cell, Ns] and (df/dlnA)^T v [cell, Nr]"""
        c, ns = len(T), n.shape[1] + 1
        X = np.zeros((ns, c))
        X[:-1] = n.T
        o = self._run([order, c], [T, P, X, v.T])
        return o[:ns * c].reshape(ns, c).T, o[ns * c:].reshape(-1, c).T

    def integrate(self, T, P, Y, dt, rtol=1e-6, atol=1e-10, cache=False, order=1):
        """T, Y [cell, Ns], the factor cache, h, status and attempts"""
        c, ns = len(T), Y.shape[1]
        o = self._run([order, c, repr(dt), repr(rtol), repr(atol), int(cache)], [T, P, Y.T])
        stride = ns * ns + 2 * ((ns + 1) // 2) + 2
        cut = np.cumsum([c, ns * c, stride * c, c, c])
        T1, Y1, C, h, st, at = np.split(o, cut)
        return T1, Y1.reshape(ns, c).T, C.reshape(c, stride), h, st.astype(int), at.astype(int)
