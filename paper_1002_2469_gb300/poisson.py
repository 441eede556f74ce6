"""The 2-D Dirichlet Poisson problem by separation of variables (Sec. 3.2 and Sec. 4).

-Laplace(u) = f on the unit square, u = 0 on the boundary, five-point stencil on a grid of
(M + 1) x (M + 1) intervals (h = 1 / (M + 1)), unknowns u[i, j] = u(x_i, y_j), i, j = 1..M, stored
as an [M, M] tensor (row i = x_i).  The orthonormal DST-I along x diagonalises the x part of the
operator; mode k = 1..M leaves one tridiagonal Toeplitz system along y,

    -v[k, j-1] + (2 + 4 sin^2(k pi / (2 (M + 1)))) v[k, j] - v[k, j+1] = h^2 fhat[k, j],

the series of Sec. 3.2 with one t_0 per mode.  All M systems are solved as one batch by the
Dichotomy kernels (the library's batched entry point); the inverse DST-I (the same transform)
returns u.  Transforms of length M + 1 = 512 to 4096, a power of two, are the library's own (64-bit fixed
point on the integer pipes); the others use torch's real FFT (cuFFT) of length M + 1 with the library's
kernels before and after it (columns transposed to rows on the way in and back on the way out).

Neumann conditions in y (bc_y="neumann"): My cell-centred unknowns y_j = (j + 1/2) / My with
du/dy = 0 at y = 0 and y = 1 (ghost cells equal to their neighbours).  Mode k then leaves the
quasi-Toeplitz system of eq. 21 (Sec. 3.1), tridiag{-1, t_0(k), -1} with
t_0(k) = 2 + (hy / hx)^2 4 sin^2(k pi / (2 (M + 1))) and psi = chi = -1 in its first and last
rows, right-hand side hy^2 fhat_k; the batch's corner step handles the two rows.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from . import _lib
from . import dichotomy as _d

__all__ = ["dst1", "mode_t0", "Poisson2D"]

# transform lengths M + 1 with the library's own fixed-point FFT; others go through torch's FFT
_FIXED = (512, 1024, 2048, 4096)


def dst1(a: torch.Tensor, dim: int = 0) -> torch.Tensor:
    """Orthonormal DST-I along `dim`: X_k = sqrt(2 / (M + 1)) sum_j a_j sin(pi j k / (M + 1)),
    j, k = 1..M.  It is its own inverse.  One real FFT of length N = M + 1 (half the padded
    length): with a_0 = a_N = 0, y_j = sin(pi j / N) (a_j + a_{N-j}) + (a_j - a_{N-j}) / 2 has
    C_k - i S_k = sum_j y_j exp(-2 pi i j k / N) with S_k = X_{2k} (the antisymmetric part) and
    C_k = X_{2k+1} - X_{2k-1} (the symmetric part, by the product-to-sum identity), so the odd
    outputs are the running sums X_{2k+1} = C_0 / 2 + C_1 + ... + C_k."""
    x = a.movedim(dim, -1)
    M = x.shape[-1]
    N = M + 1
    z = torch.zeros(x.shape[:-1] + (1,), dtype=x.dtype, device=x.device)
    xp = torch.cat([z, x], dim=-1)                       # a_j, j = 0..N-1
    xr = torch.cat([z, x.flip(-1)], dim=-1)              # a_{N-j}
    s = torch.sin(torch.arange(N, dtype=x.dtype, device=x.device) * (math.pi / N))
    y = s * (xp + xr) + 0.5 * (xp - xr)
    Y = torch.fft.rfft(y, dim=-1)
    out = torch.empty_like(x)
    out[..., 1::2] = -Y.imag[..., 1:1 + M // 2]            # X_{2m}, m = 1..M/2
    C = Y.real
    odd = torch.cumsum(C, dim=-1) - 0.5 * C[..., :1]       # X_{2m+1}, m = 0..(M-1)/2
    out[..., 0::2] = odd[..., :(M + 1) // 2]
    return (out * math.sqrt(2.0 / N)).movedim(-1, dim).contiguous()


def mode_t0(M: int) -> np.ndarray:
    """t_0 of the tridiagonal system of mode k = 1..M: 2 + 4 sin^2(k pi / (2 (M + 1)))."""
    k = np.arange(1, M + 1, dtype=np.float64)
    return 2.0 + 4.0 * np.sin(k * math.pi / (2.0 * (M + 1))) ** 2


def _transform_table(N: int) -> np.ndarray:
    """The table of dichotomy_dst: N twiddles and N / 2 + 1 sines as 64-bit fractions (from extended
    precision, at least 64 bits on both x86 and AArch64 hosts)."""
    pi = np.longdouble("3.14159265358979323846264338327950288")
    quarter = np.sin(np.arange(N // 4 + 1, dtype=np.longdouble) * (2 * pi / N))     # sin 2 pi m / N, a quarter
    m = np.arange(N)
    r = m % (N // 2)
    sin = np.where(m < N // 2, 1, -1) * quarter[np.minimum(r, N // 2 - r)]
    cos = sin[(m + N // 4) % N]
    sine = np.sin(np.arange(N // 2 + 1, dtype=np.longdouble) * (pi / N))
    w = np.concatenate([np.stack([(cos + 1) / 2, (1 - sin) / 2], axis=1).ravel(), sine])
    one = w >= 1
    words = np.where(one, np.longdouble(0), w * np.longdouble(2.0 ** 64)).astype(np.uint64)
    words[one] = np.uint64(0xFFFFFFFFFFFFFFFF)
    words[:2 * N] &= np.uint64(0xFFFFFFFFFFFFFFFE)                                   # twiddle words are even
    return words


class Poisson2D:
    """Solver for an [M, My] grid (My = M by default): Dirichlet in x; Dirichlet (My interior
    nodes, hy = 1 / (My + 1)) or Neumann (My cell centres, hy = 1 / My) in y.  The batch of M
    mode systems is planned once."""

    def __init__(self, M: int, precision: int = _d.PREC_AUTO, device=None, My: int | None = None,
                 bc_y: str = "dirichlet"):
        self.M = int(M)
        self.My = int(My) if My is not None else self.M
        if bc_y not in ("dirichlet", "neumann"):
            raise ValueError("bc_y must be 'dirichlet' or 'neumann'")
        self.bc_y = bc_y
        self.hx = 1.0 / (self.M + 1)
        self.hy = 1.0 / (self.My + 1) if bc_y == "dirichlet" else 1.0 / self.My
        self.h = self.hy
        k = np.arange(1, self.M + 1, dtype=np.float64)
        t0 = 2.0 + (self.hy / self.hx) ** 2 * 4.0 * np.sin(k * math.pi / (2.0 * (self.M + 1))) ** 2
        ones = np.ones(self.M)
        corners = dict(psi=-ones, chi=-ones) if bc_y == "neumann" else {}
        self.batch = _d.Batch(np.full(self.M, self.My, dtype=np.int64), -ones, t0, -ones, precision=precision,
                              **corners)
        self.device = device
        # coefficients of the transforms' first step, for the right-hand side (with hy^2) and the modes
        N = self.M + 1
        s = np.sin(np.arange(N // 2 + 1) * (math.pi / N))
        self._table = None
        if N in _FIXED:
            words = _transform_table(N)
            dev = self.batch.workspace.device
            self._table = torch.from_numpy(words.view(np.int64)).to(dev)
            self._scale = 0.5 * math.sqrt(2.0 / N)
            return
        c = np.stack([s + 0.5, s - 0.5], axis=1) * math.sqrt(2.0 / N)
        dev = self.batch.workspace.device
        self._coef_f = torch.from_numpy(c * (self.hy * self.hy)).to(dev)
        self._coef_v = torch.from_numpy(c).to(dev)

    def _dst(self, a: torch.Tensor, factor: float) -> torch.Tensor:
        """The orthonormal DST-I of a contiguous [M, My] array along its first axis, times factor (1 or hy^2)."""
        L, stream = _lib.load(), _d._stream(None)
        if self._table is not None:
            out = torch.empty_like(a)
            work = torch.empty((self.My + 1) // 2 * 2 * (self.M + 1), dtype=torch.float64, device=a.device)
            _lib.check(L.dichotomy_dst(self.M, self.My, _d._dev(a, "f"), self._table.data_ptr(), self._scale * factor,
                                       work.data_ptr(), out.data_ptr(), stream), "dichotomy_dst")
            return out
        coef = self._coef_v if factor == 1.0 else self._coef_f
        z = torch.empty((self.My, self.M + 1), dtype=torch.float64, device=a.device)
        _lib.check(L.dichotomy_dst_rows_pre(self.M, self.My, _d._dev(a, "f"), coef.data_ptr(), z.data_ptr(), stream),
                   "dichotomy_dst_rows_pre")
        Z = torch.fft.rfft(z, dim=-1)
        out = torch.empty_like(a)
        _lib.check(L.dichotomy_dst_rows_post(self.M, self.My, Z.data_ptr(), out.data_ptr(), stream), "dichotomy_dst_rows_post")
        return out

    def solve(self, f: torch.Tensor) -> torch.Tensor:
        """u for the right-hand side f ([M, My], float64, CUDA)."""
        if f.shape != (self.M, self.My):
            raise ValueError(f"f must be [{self.M}, {self.My}]")
        rhs = self._dst(f.detach().contiguous(), self.hy * self.hy)    # [k, j]: mode k along y
        v = self.batch.solve(rhs.reshape(-1)).reshape(self.M, self.My)
        return self._dst(v, 1.0)

    def status(self) -> int:
        return self.batch.status()
