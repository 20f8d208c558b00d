"""Sensor noise on rendered images (Sec. III.C): Poisson photon shot noise
plus Gaussian read noise, computed by libosog's osog_sensor_noise."""
from __future__ import annotations

import torch

from . import _lib
from ._lib import check
from ._stream import raw_stream


def sensor_noise(image: torch.Tensor, photons_per_unit: float, read_sigma: float, seed: int,
                 out: torch.Tensor | None = None) -> torch.Tensor:
    """(Poisson(g max(I, 0)) + read_sigma N(0, 1)) / g elementwise, with a
    counter-based generator keyed by seed (reproducible per element)."""
    if image.device.type != "cuda" or image.dtype != torch.float32 or not image.is_contiguous():
        raise ValueError("image must be a contiguous CUDA float32 tensor")
    if out is None:
        out = torch.empty_like(image)
    check(_lib.lib().osog_sensor_noise(image.data_ptr(), image.numel(),
                                       float(photons_per_unit), float(read_sigma),
                                       int(seed) & 0xFFFFFFFFFFFFFFFF, out.data_ptr(),
                                       raw_stream(image.device.index)),
          "osog_sensor_noise")
    return out
