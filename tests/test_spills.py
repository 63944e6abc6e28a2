"""The phase-field collision of pairs keeps its values in registers: spilled, a box with a gradient at
most nodes took longer than the tiled step (FP32, D3Q19)."""
import os
import re
import subprocess

from paper_1602_07483_gb300 import build


def test_phi_pairs_do_not_spill(tmp_path):
    out = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", "-o", str(tmp_path / "o.o"),
                         os.path.join(build.CSRC, "kern_pair_f32.cu")], capture_output=True, text=True, check=True).stderr
    found = {}
    for part in out.split("Compiling entry function ")[1:]:
        name = re.match(r"'(\S+)'", part).group(1)
        found[name] = [int(v) for v in re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", part).groups()]
    phi = {n: v for n, v in found.items() if "k_phi_pair" in n}
    assert len(phi) == 5  # one per lattice
    assert all(v == [0, 0] for v in phi.values()), phi
