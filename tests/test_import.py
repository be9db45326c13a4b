"""The package imports on a torch that lacks the private functions its calls are faster with."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_import_without_the_raw_stream_function():
    code = ("import torch\n"
            "if hasattr(torch._C, '_cuda_getCurrentRawStream'): del torch._C._cuda_getCurrentRawStream\n"
            "import paper_2409_19156_gb300 as zp\n"
            "from paper_2409_19156_gb300 import inputs\n"
            "assert len(inputs.radial_modes(4)[0]) == 9 and callable(zp.radial)\n")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)
