"""CPU: the block-sparse order search of the library on host data alone (a small program around its source):
charges in wide steps give the order that charges in steps of one give, and cost no array over their range;
tensors whose symmetries differ get an order (their contraction is refused later)."""
import os
import subprocess

import pytest

from paper_2401_01921_gb300 import build

PROGRAM = r"""
#include "tnx_network.cpp"
#include <chrono>
#include <cstdio>
#include <cstdlib>

// nsec sectors of charges (s - nsec / 2) * step; a second charge takes -step, 0 or step times that
static BondD bond(int dir, int nsym, int nsec, int step, int deg) {
  BondD b;
  b.dir = nsym ? dir : TNX_BD_REG;
  b.nsym = nsym;
  b.kinds.assign(nsym, TNX_U1);
  b.zn.assign(nsym, 0);
  b.nsec = nsec;
  for (int s = 0; s < nsec; ++s) {
    for (int c = 0; c < nsym; ++c) b.qn.push_back((s - nsec / 2) * step * (c ? s % 3 - 1 : 1));
    b.deg.push_back(deg + s);
  }
  b.finish();
  return b;
}

// argv: symmetries, step between charges, sectors of the virtual bonds, symmetries of tensor 0 (if others);
// prints the order and the shortest time in ms
int main(int argc, char** argv) {
  const int nsym_all = atoi(argv[1]), step = atoi(argv[2]), nsec = atoi(argv[3]);
  const int nsym_0 = argc > 4 ? atoi(argv[4]) : nsym_all;
  const char* name[5] = {"L", "psi", "W1", "W2", "R"};
  const char* labels[5] = {"a,w0,ap", "a,s1,s2,b", "w0,s1p,s1,w1", "w1,s2p,s2,w2", "b,w2,bp"};
  double best = 1e30;
  std::string order;
  for (int r = 0; r < 5; ++r) {
    tnx_network& net = *new tnx_network();   // left alive: its destructor wants a context
    std::map<std::string, int> seen;
    for (int i = 0; i < 5; ++i) {
      NetTensor t;
      t.name = name[i];
      t.labels = split_labels(labels[i]);
      t.t = new tnx_tensor();
      const int nsym = i ? nsym_all : nsym_0;
      for (const std::string& l : t.labels) {
        const bool chi = l[0] == 'a' || l[0] == 'b';
        t.t->bonds.push_back(bond(seen[l]++ ? TNX_BD_OUT : TNX_BD_IN, nsym, !nsym ? 1 : chi ? nsec : l[0] == 'w' ? 3 : 2,
                                  step, chi ? 10 : 1));
        t.perm.push_back((int)t.perm.size());
      }
      t.t->rank = (int)t.t->bonds.size();
      net.ts.push_back(t);
    }
    const auto t0 = std::chrono::steady_clock::now();
    sparse_optimal_tree(&net);
    best = std::min(best, std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count());
    order = tree_string(&net, net.root);
  }
  printf("%s %.6f\n", order.c_str(), best);
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    lib = build.build()
    d = tmp_path_factory.mktemp("order")
    (d / "search.cpp").write_text(PROGRAM)
    exe = str(d / "search")
    subprocess.run([build._nvcc(), "-x", "cu", "-O3", "-std=c++17", str(d / "search.cpp"), "-o", exe,
                    f"-I{build.INCLUDE}", f"-I{build.CSRC}", *build.ARCH, f"-L{os.path.dirname(lib)}", "-l:libtnx.so",
                    "-Xlinker", f"-rpath={os.path.dirname(lib)}"], check=True, capture_output=True)

    def run(*args):
        order, ms = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout.split()
        return order, float(ms)
    return run


# ranges of keys inside and beyond the array's limit, one and two charges
@pytest.mark.parametrize("nsym,step,nsec", [(1, 1000, 20), (1, 20000, 20), (1, 30000, 8), (2, 60, 20), (2, 400, 6)])
def test_wide_charges(search, nsym, step, nsec):
    order, ms = search(nsym, step, nsec)
    ref, ref_ms = search(nsym, 1, nsec)
    assert order == ref
    assert ms <= 20 * ref_ms + 5.0   # an array over the range took 100 to 270 times as long for one charge


@pytest.mark.parametrize("nsym,nsym0", [(1, 0), (0, 1), (2, 1), (1, 2)])
def test_tensors_of_different_symmetries(search, nsym, nsym0):
    """Such a network is refused when it is launched; the search before that has to survive it."""
    order, _ = search(nsym, 1, 8, nsym0)
    assert sorted(order.replace("(", "").replace(")", "").split(",")) == ["L", "R", "W1", "W2", "psi"]
