"""Streaming local solves: FP64 factors, and several handles at once."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FP64_SCRIPT = """
import sys
import numpy as np, torch
from oracle import a2ls_oracle as O
from paper_2201_02250_gb300 import a2ls
from workloads import pde
m, nb, overlap, variant, pou, kernel = (int(v) if v.lstrip('-').isdigit() else v for v in sys.argv[1:7])
prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=overlap, nev=3)
P, keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, prob.nev, variant=variant, pou=pou)
assert P.tuning()["local_solve_threads"] == kernel, P.tuning()
ref = O.setup(prob.A, prob.part, prob.overlap, prob.nev, pou=pou)
P.set_coarse_basis(ref.coarse.W)
r = torch.as_tensor(prob.b, device="cuda")
z = torch.empty_like(r)
P.apply(r, z)
torch.cuda.synchronize()
want = O.apply(ref, prob.b, variant)
err = np.linalg.norm(z.cpu().numpy() - want) / np.linalg.norm(want)
assert err < 1e-10, err
"""


@pytest.mark.parametrize("m,nb,overlap,variant,pou", [
    (13, 2, 0, "ras", "boolean"),             # one ragged block per subdomain, no overlap
    (16, 2, 1, "deflated_ras", "boolean"),    # 64 + 16 rows: a full block and a short one
    (31, 2, 2, "deflated_asm", "multiplicity"),
    (72, 3, 2, "deflated_ras", "multiplicity"),   # several panel chunks a block
])
@pytest.mark.parametrize("kernel", [3000, 3004, 3008])
def test_fp64_streaming_matches_oracle(tmp_path, m, nb, overlap, variant, pou, kernel):
    """The FP64 apply with each streaming shape, chosen through a saved autotune file, to the FP64 apply's bound
    of 1e-10."""
    from workloads import pde
    from oracle import a2ls_oracle as O
    prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=overlap, nev=3)
    sizes = [s.n_i for s in O.overlapping_subdomains(prob.A, prob.part, prob.overlap)]
    mode = (0 if pou == "boolean" else 1) if variant.endswith("ras") else 2
    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({f"local_solve4_fp64_N{nb * nb}_max{max(sizes)}_mode{mode}": kernel}))
    env = dict(os.environ, A2LS_AUTOTUNE_CACHE=str(cache))
    r = subprocess.run([sys.executable, "-c", FP64_SCRIPT, str(m), str(nb), str(overlap), variant, pou, str(kernel)],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("kernel", [3000, 3004, 3008])
@pytest.mark.parametrize("first,second", [((96, 3), (20, 2)), ((20, 2), (96, 3)), ((60, 2), (45, 2))])
def test_handles_of_different_sizes_side_by_side(kernel, first, second):
    """A handle's streaming solves still launch after another handle, whose largest subdomain needs another
    amount of shared memory, has been set up, and give the same values as before."""
    import torch
    from paper_2201_02250_gb300 import a2ls
    from workloads import pde
    out = []
    handles = []
    for m, nb in (first, second):
        prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=1, nev=3)
        P, keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, prob.nev, precision="fp32",
                                  local_solve_kernel=kernel)
        r = torch.as_tensor(prob.b, device="cuda")
        z = torch.empty_like(r)
        P.apply(r, z)
        torch.cuda.synchronize()
        handles.append((P, keep, r))
        out.append(z.clone())
    for (P, _, r), want in zip(handles, out):
        z = torch.empty_like(r)
        P.apply(r, z)
        torch.cuda.synchronize()
        assert np.array_equal(z.cpu().numpy(), want.cpu().numpy())


FOOTPRINT_SCRIPT = """
import sys
import torch
from paper_2201_02250_gb300 import a2ls
from workloads import pde
prob = pde.tiny_conv_diff(m=300, nb=5, overlap=1, nev=0)
P, keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, 0, variant="ras", local_solve_kernel=int(sys.argv[1]))
P.solve(torch.as_tensor(prob.b, device="cuda"), torch.zeros(prob.n, dtype=torch.float64, device="cuda"), 1e-1,
        allow_not_converged=True)
a2ls.trim_memory()
free, total = torch.cuda.mem_get_info()
print(P.tuning()["local_solve_threads"], total - free, max(len(a) + len(b) for a, b in P.subdomains()))
"""


def test_fp64_factors_are_held_once_unless_streamed(tmp_path):
    """What the device holds for a handle of 25 subdomains of 3600 rows (band 60, so that a second copy of the factors
    is 2 x 90000 x 60 doubles and more): a kernel known to be faster than the streaming one leaves none behind."""
    copy = 2 * 90000 * 60 * 8

    def footprint(option, cached=None):
        cache = tmp_path / f"tune{option}_{cached}.json"
        cache.write_text("{}" if cached is None else json.dumps({f"local_solve4_fp64_N25_max{rows}_mode0": cached}))
        r = subprocess.run([sys.executable, "-c", FOOTPRINT_SCRIPT, str(option)], cwd=ROOT, capture_output=True, text=True,
                           env=dict(os.environ, A2LS_AUTOTUNE_CACHE=str(cache)), timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return [int(v) for v in r.stdout.split()]

    kernel, base, rows = footprint(512)
    assert kernel == 512
    kernel, held, _ = footprint(0, 512)
    assert kernel == 512 and held - base < copy // 2
    kernel, held, _ = footprint(0, 3000)
    assert kernel == 3000 and held - base > copy // 2


def test_fp64_copy_is_withheld_and_given_back(tmp_path):
    from paper_2201_02250_gb300 import _build
    exe, libdir = str(tmp_path / "stream_memory"), os.path.dirname(_build.LIB)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    os.path.join(ROOT, "tests", "cpp", "stream_memory.cu"), "-L", libdir, "-lA2LS", "-Xlinker", "-rpath=" + libdir,
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
