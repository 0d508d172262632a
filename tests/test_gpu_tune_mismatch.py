"""A tuning-cache line that names a kernel of the other precision is passed over: the apply runs its default kernel
and matches the oracle (1e-5 of the norm in complex64, 1e-12 in complex128)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = '''
import sys; sys.path.insert(0, %r)
import numpy as np, torch
import paper_2606_03599_gb300 as pc
from oracle import oracle as O
from workloads import complex_gaussian, two_phase_sphere
N, dt = 12, sys.argv[1]
cell = two_phase_sphere(N, 0.35, 3)
h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
C0, rho0, L = pc.pc_grid_units(h)
pb = O.problem_from_cell(cell, C0=C0, rho0=rho0, L=L)
pc.pc_set_k(h, (0.2, 0.3, 0.1))
x = complex_gaussian((3, N ** 3), 4)[:, O.block_index((N,) * 3, 2)]
if dt == "c64": x = x.astype(np.complex64)
d = torch.from_numpy(np.ascontiguousarray(x)).reshape(-1).cuda(); y = torch.zeros_like(d)
pc.pc_block_apply(h, 2, d, y, shift=0.7)
print(pc.pc_tuned_config(h, pc.PC_C64 if dt == "c64" else pc.PC_C128, 0, 1)[:2])
ref = O.apply_block(pb, (0.2, 0.3, 0.1), 2, x.astype(complex), 0.7).reshape(-1)
print(np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref))
''' % ROOT


@pytest.mark.parametrize("dtype,shape,tol", [("c64", 8, 1e-5), ("c128", 9, 1e-12)])
def test_a_kernel_of_the_other_precision_is_passed_over(tmp_path, dtype, shape, tol):
    import torch
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    path = tmp_path / "tune.json"
    path.write_text('"6,6,12,%s,blocks,phase,cubic,n1,sm%d": {"kind": 0, "shape": %d, "tz": 2, "ctas": 6, "us": 1}\n'
                    % (dtype, sm, shape))
    out = subprocess.run([sys.executable, "-c", CODE, dtype], env=dict(os.environ, PC_TUNE_CACHE=str(path)),
                         capture_output=True, text=True, check=True).stdout.split("\n")
    assert out[0] == ("(0, 9)" if dtype == "c64" else "(0, 8)")
    assert float(out[1]) <= tol
