"""The host-side calls with a PyTorch that was built without CUDA."""
import subprocess
import sys


def test_import_and_model_files_without_cuda_bindings():
    code = ("import torch\n"
            "del torch._C._cuda_getCurrentRawStream\n"
            "import numpy as np\n"
            "import paper_1512_06473_gb300 as q\n"
            "blob = q.serialize_model([{'kind': 'fc', 'D': np.zeros((2, 4, 2), np.float32),\n"
            "                           'codes': np.zeros((2, 3), np.uint8)}], (4, 1, 1))\n"
            "assert q.model_info(blob)[0] == 1\n")
    subprocess.run([sys.executable, "-c", code], check=True, timeout=600)
