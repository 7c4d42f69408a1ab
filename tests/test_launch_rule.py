"""Which marches launch their kernels as programmatic dependents: the rule of mot_internal.cuh,
compiled alone (host code, no device needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "mot_internal.cuh"
#include <cstdio>
using mot::MarchScope;
using mot::dependent_launches;
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    mot_ctx owner, a, b, other;
    a.shared_src = b.shared_src = &owner;
    owner.n_shared = 2;
    {   // a borrower that marches alone (the adjoint march of the gradient)
        MarchScope m(&a);
        CHECK(dependent_launches(&a));
        {   // the owner beside it, and another setup's march
            MarchScope n(&owner), o(&other);
            CHECK(!dependent_launches(&a) && !dependent_launches(&owner));
            CHECK(dependent_launches(&other));
        }
        CHECK(dependent_launches(&a));
    }
    {   // several right-hand sides in one call
        MarchScope m(&owner, 0), n(&a, 0), o(&b, 0);
        CHECK(!dependent_launches(&owner) && !dependent_launches(&a) && !dependent_launches(&b));
    }
    {   // a graph's launches stay of one kind
        MarchScope m(&a, 0), n(&other, 1);
        CHECK(!dependent_launches(&a) && dependent_launches(&other));
    }
    CHECK(owner.marching.load() == 0 && other.marching.load() == 0);
    CHECK(dependent_launches(&owner) && dependent_launches(&b));
    return 0;
}
"""


def test_dependent_launches_follow_the_call(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "rule.cu"
    src.write_text(SOURCE)
    exe = tmp_path / "rule"
    inc = [os.path.join(ROOT, "include"), os.path.join(ROOT, "paper_2407_03323_gb300", "csrc")]
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", inc[0],
                        "-I", inc[1], str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
