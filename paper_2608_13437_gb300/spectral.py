"""Spectral diagnostics on the device (Sec. 3.2): Eq. 7's dissipation rates with curl
and divergence taken spectrally (torch.fft, i.e. cuFFT) and mu_local applied per cell in
physical space, and the shell-averaged kinetic-energy spectrum normalised so that
sum_k E(k) = <|u|^2> / 2. Inputs are the primitive fields that lbm_moments(LBM_MOM_PRIM)
writes (rho, u_x, u_y, u_z, T, p), as a device tensor (6, nz, ny, nx), on a periodic box
of side L_box per axis.

FP64 tensors on the GPU take the passes of lbm_spectral.h: curl and divergence are formed
in spectral space (four fields instead of nine gradients), and a complex transform carries
two real fields, so a sample takes one complex and one real transform forward and two
complex ones back, and one pass for the means. The FP64 rate bounds the transforms on
this part (364 us for a complex one at 128^3), so their number counts. Other tensors
(CPU, FP32, under autograd or a functional transform) take plain tensor operations.
"""
from __future__ import annotations

import math

T_SUTHERLAND = 0.4042
_DOUBLES = 2 + 2 * 1216  # LBM_SPECTRAL_DOUBLES
_MOST_SHELLS = 6000


def _on_device(t):
    """Whether the tensor's values alone are wanted and the library's passes can read it: a
    plain FP64 CUDA tensor, nothing recording, transforming or capturing operations."""
    import torch
    from torch.autograd import forward_ad
    if (type(t) is not torch.Tensor or not t.is_cuda or t.dtype != torch.float64
            or (t.requires_grad and torch.is_grad_enabled()) or not 0 < t.numel() < 1 << 31):
        return False
    peek = getattr(torch._C._functorch, "peek_interpreter_stack", None)
    return not (torch.compiler.is_compiling() or peek is None or peek() is not None
                or getattr(forward_ad, "_current_level", -1) >= 0
                or torch._C._len_torch_dispatch_stack()
                or torch.cuda.is_current_stream_capturing())


def _numbers(*values):
    return all(isinstance(v, (int, float)) for v in values)


def _sizes(*values):
    """Whether these are the positive numbers that the library's passes divide by; what any
    other value gives or raises is left to the tensor operations."""
    return _numbers(*values) and all(1e-300 < v < 1e300 for v in values)


def _k(n, L_box, device, dtype):
    import torch
    k = torch.fft.fftfreq(n, d=L_box / n, device=device, dtype=dtype) * (2 * math.pi)
    if n % 2 == 0:  # no derivative of the Nyquist mode of a real field
        k[n // 2] = 0.0
    return k


def gradients(u, L_box=2 * math.pi):
    """g[a][b] = d_a u_b (3, 3, nz, ny, nx) for u (3, nz, ny, nx)."""
    import torch
    nz, ny, nx = u.shape[1:]
    dt = u.dtype
    kx = _k(nx, L_box, u.device, dt).view(1, 1, nx)
    ky = _k(ny, L_box, u.device, dt).view(1, ny, 1)
    kz = _k(nz, L_box, u.device, dt).view(nz, 1, 1)
    uh = torch.fft.fftn(u, dim=(1, 2, 3))
    out = torch.empty((3, 3) + tuple(u.shape[1:]), dtype=dt, device=u.device)
    for a, k in enumerate((kx, ky, kz)):
        out[a] = torch.fft.ifftn(1j * k * uh, dim=(1, 2, 3)).real
    return out


def dissipation(prim, mu, T_ref, sutherland, rho_ref, L_box=2 * math.pi):
    """(eps_s, eps_d) of Eq. 7 from primitive fields (6, nz, ny, nx) (FP64 recommended)."""
    import torch
    if (prim.ndim == 4 and len(prim) >= 5 and _numbers(mu, T_ref) and _sizes(rho_ref, L_box)
            and (not sutherland or _sizes(T_ref)) and _on_device(prim)):
        return _dissipation_device(prim, mu, T_ref, sutherland, rho_ref, L_box)
    g = gradients(prim[1:4], L_box)
    wx, wy, wz = g[1, 2] - g[2, 1], g[2, 0] - g[0, 2], g[0, 1] - g[1, 0]
    div = g[0, 0] + g[1, 1] + g[2, 2]
    T = prim[4]
    if sutherland:
        t = T / T_ref
        m = mu * (1 + T_SUTHERLAND) * t ** 1.5 / (t + T_SUTHERLAND)
    else:
        m = torch.full_like(T, mu)
    eps_s = torch.mean(m * (wx * wx + wy * wy + wz * wz)) / rho_ref
    eps_d = 4.0 / 3.0 * torch.mean(m * div * div) / rho_ref
    return float(eps_s), float(eps_d)


def _packed_spectra(u):
    """Spectrum of u_x + i u_y over the whole grid and half spectrum of u_z."""
    import torch
    return (torch.fft.fftn(torch.complex(u[0], u[1])).contiguous(),
            torch.fft.rfftn(u[2]).contiguous())


def _dissipation_device(prim, mu, T_ref, sutherland, rho_ref, L_box):
    import torch

    from . import lbm
    nz, ny, nx = prim.shape[1:]
    with torch.cuda.device(prim.device):
        L, stream = lbm.lib(), torch.cuda.current_stream().cuda_stream
        zh, ch = _packed_spectra(prim[1:4])
        wh = zh.new_empty((2, nz, ny, nx))
        lbm.check(L.lbm_spectral_curl_div(zh.data_ptr(), ch.data_ptr(), wh.data_ptr(), nx, ny, nz,
                                          2 * math.pi / L_box, stream))
        w = torch.fft.ifftn(wh, dim=(1, 2, 3), norm="forward").contiguous()
        T = prim[4].contiguous().resolve_neg()  # its values are read, whatever view it is
        out = torch.empty(_DOUBLES, dtype=torch.float64, device=prim.device)
        lbm.check(L.lbm_spectral_dissipation(w.data_ptr(), T.data_ptr(), nx * ny * nz, mu, T_ref,
                                             int(bool(sutherland)), out.data_ptr(), stream))
        s, d = out[:2].tolist()
    return s / rho_ref, 4.0 / 3.0 * d / rho_ref


def energy_spectrum(u, L_box=2 * math.pi):
    """(k, E(k)) over unit-width shells of |k| L; sum(E) = <|u|^2> / 2."""
    import torch
    nz, ny, nx = u.shape[1:]
    if u.is_cuda and _numbers(L_box) and not 0 < L_box < math.inf:
        # No shells: of a negative side the tensor operations would use negative indices, which
        # a kernel cannot report; of the others all shells are NaN, of which the GPU makes the
        # lowest integer and PyTorch a RuntimeError.
        raise (IndexError if L_box < 0 else RuntimeError)(f"L_box must be positive and finite, not {L_box}")
    # the shells' pass adds in any order, so runs that ask for the same bits every time take
    # the tensor operations, which give them
    if (u.ndim == 4 and len(u) == 3 and _sizes(L_box) and _on_device(u)
            and not torch.are_deterministic_algorithms_enabled()):
        from . import lbm
        L = lbm.lib()
        shells = L.lbm_spectral_shell_count(nx, ny, nz)
        if shells <= _MOST_SHELLS:
            with torch.cuda.device(u.device):
                zh, ch = _packed_spectra(u)
                e = torch.zeros(shells, dtype=u.dtype, device=u.device)
                lbm.check(L.lbm_spectral_shells(zh.data_ptr(), ch.data_ptr(), nx, ny, nz, e.data_ptr(),
                                                shells, torch.cuda.current_stream().cuda_stream))
                return torch.arange(shells, device=u.device), e
    dt = u.dtype
    kx = _k_full(nx, L_box, u.device, dt).view(1, 1, nx)
    ky = _k_full(ny, L_box, u.device, dt).view(1, ny, 1)
    kz = _k_full(nz, L_box, u.device, dt).view(nz, 1, 1)
    kmag = torch.sqrt(kx * kx + ky * ky + kz * kz) * (L_box / (2 * math.pi))
    shell = torch.round(kmag).to(torch.int64).reshape(-1)
    n = nx * ny * nz
    e = torch.zeros(int(shell.max()) + 1, dtype=dt, device=u.device)
    for b in range(3):
        uh = torch.fft.fftn(u[b]) / n
        e.index_add_(0, shell, (0.5 * uh.abs() ** 2).reshape(-1))
    return torch.arange(len(e), device=u.device), e


def _k_full(n, L_box, device, dtype):
    import torch
    return torch.fft.fftfreq(n, d=L_box / n, device=device, dtype=dtype) * (2 * math.pi)
