"""heat_step with an infinite time step on an unshifted hierarchy: u / dt is 0, so
the step is a steady solve (theta = 1: A u = b1; theta = 1/2: A (u + u_old) =
b1 + b0).  On the host: quotients by an infinite divisor are those of division.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.sparse.linalg as spla

import eb_inputs as ei
from oracle import eb as oeb

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_06083_gb300", "csrc")

PROG = r"""
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <limits>
#include "divide.cuh"
template <class A>
static int bad() {
  const A inf = std::numeric_limits<A>::infinity(), max = std::numeric_limits<A>::max();
  const ebk::DivBy<A> c = ebk::DivBy<A>::of((double)inf);
  int n = 0;
  for (A a : {(A)0, (A)1, (A)-3.5e10, max, -max, inf, -inf, (A)std::nan("")}) {
    const A want = a / inf, got = ebk::div_by(a, c);
    if (!(got == want || (std::isnan(got) && std::isnan(want)))) ++n;
  }
  return n;
}
int main() {
  std::printf("%d\n", bad<double>() + bad<float>());
  return 0;
}
"""


def test_quotients_by_infinity(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(PROG)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-I", HDR, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    assert int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("theta", [1.0, 0.5])
def test_infinite_time_step(theta):
    import torch
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid, ls = ei.circle_k1(130)
    h = eb.EB(grid, ls)
    ref = oeb.build(grid, ls)
    amg = eb.AMG(h, 0.0)
    rng = np.random.default_rng(3)
    b1, b0, u0 = (rng.standard_normal(ref.num_cp) for _ in range(3))
    u = torch.tensor(ref.to_grid(u0), device="cuda")
    st = amg.heat_step(u, torch.tensor(ref.to_grid(b1), device="cuda"), float("inf"), theta,
                       torch.tensor(ref.to_grid(b0), device="cuda"), rtol=1e-13)
    assert st.converged
    want = spla.spsolve(ref.A.tocsc(), b1) if theta == 1.0 else spla.spsolve(ref.A.tocsc(), b1 + b0) - u0
    got = ref.from_grid(u.cpu().numpy())
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
