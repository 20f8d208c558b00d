"""The current CUDA stream's handle, for the C ABI's stream arguments."""
from __future__ import annotations

import torch


def raw_stream(index: int | None = None) -> int:
    """Handle of the current CUDA stream of device `index` (default: the
    current device) of a process that has used CUDA, without a
    torch.cuda.Stream object around it (3 us of a 30 us call)."""
    return torch._C._cuda_getCurrentRawStream(
        torch._C._cuda_getDevice() if index is None else index)
