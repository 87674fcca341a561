"""The package imports with a torch that lacks the private stream accessor (builds without CUDA), and the calls then take the
current stream from torch's public interface."""
import subprocess
import sys

CODE = """
import torch
if hasattr(torch._C, "_cuda_getCurrentRawStream"):
    del torch._C._cuda_getCurrentRawStream
import paper_2505_13254_b200.step
from paper_2505_13254_b200 import binding
class Stream:
    cuda_stream = 0x1234
torch.cuda.current_stream = lambda device: Stream() if device == 3 else None
assert binding._raw_stream(3) == 0x1234
"""


def test_the_private_stream_accessor_is_optional():
    subprocess.run([sys.executable, "-c", CODE], check=True)
