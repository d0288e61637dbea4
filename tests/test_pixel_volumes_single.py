"""Single-precision volumes of pixel triples, as the pixelised 4pCF kernel forms
them (cross product, then dot product): over every ordered triple of the 256
pixels the value is below the kernel's threshold 2e-5 exactly when the FP64
volume is below 1e-9, and has its sign otherwise. Covers every order in which
the kernel takes the three spokes and both signs of the first."""
import numpy as np


def test_every_pixel_triple():
    p = np.arange(256)
    z = (2.0 * (p >> 4) + 1.0) / 16.0 - 1.0
    phi = np.pi * (2.0 * (p & 15) + 1.0) / 16.0
    rho = np.sqrt((1.0 - z) * (1.0 + z))
    u = np.stack([rho * np.cos(phi), rho * np.sin(phi), z], axis=1)
    v = u.astype(np.float32)
    for i in range(256):
        n64 = np.cross(np.broadcast_to(u[i], u.shape), u)
        V64 = n64 @ u.T
        a, b = v[i], v
        n32 = np.stack([a[1] * b[:, 2] - a[2] * b[:, 1], a[2] * b[:, 0] - a[0] * b[:, 2],
                        a[0] * b[:, 1] - a[1] * b[:, 0]], axis=1)
        V32 = (n32[:, None, 0] * v[None, :, 0] + n32[:, None, 1] * v[None, :, 1]
               + n32[:, None, 2] * v[None, :, 2])
        assert V32.dtype == np.float32
        degenerate = np.abs(V64) < 1e-9
        assert np.array_equal(np.abs(V32) < np.float32(2e-5), degenerate)
        assert np.array_equal(np.sign(V32)[~degenerate], np.sign(V64)[~degenerate])
        assert np.abs(V32 - V64).max() < 2e-6  # the bound the threshold rests on
