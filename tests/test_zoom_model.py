"""CPU model of the band-limited inverse FFT by output residues (csrc/zoom.cuh):
the tables, slots and twiddle indices of the kernel, pass by pass in numpy,
against the plain inverse DFT of the zero-extended band."""
import numpy as np
import pytest


def w(L, i):
    """exp(2 pi i i / L), the index reduced first as the kernel's table look-ups are."""
    return np.exp(2j * np.pi * (np.asarray(i) % L) / L)


def zoom_columns(Y, b0, M, N, QA, QB, QC, P, residues):
    """Outputs {t: value} of the given residues of one row, with the kernel's slots and indices."""
    B, QP = len(Y), QB * QC
    Q = QA * QP
    R = M // Q
    assert R * Q == M and B <= Q and N % M == 0
    QAP = (QA | 1) if P < 16 else QA
    G = len(residues)
    assert G <= P
    Yq = np.zeros(Q, complex)
    for j in range(Q):
        u = j - b0 % Q
        u += Q if u < 0 else 0
        if u < B:
            Yq[j] = Y[u]
    E = np.zeros((2, QA, P), complex)
    for t in range(2):
        for p in range(QA):
            base = b0 // QP + t
            g = p - base % QA
            g = (g + QA if g < 0 else g) + base
            for col, r in enumerate(residues):
                kap = QP * g % M
                assert kap * r < 2 ** 32
                E[t, p, col] = w(M, kap * r)
    tile = np.full(QP * QAP * P, np.nan, complex)
    for b in range(QP):
        for col in range(G):
            e = E[1 if b < b0 % QP else 0, :, col]
            v = Yq[b + QP * np.arange(QA)] * e
            v = np.fft.ifft(v) * QA
            tile[b * QAP * P + col + P * np.arange(QA)] = v
    if QC > 1:
        for b1 in range(QC):
            for k1 in range(QA):
                for col, r in enumerate(residues):
                    at = (b1 * QAP + k1) * P + col + QC * QAP * P * np.arange(QB)
                    i = QC * (r + R * k1)
                    assert i < M
                    tile[at] = np.fft.ifft(tile[at] * w(M, i) ** np.arange(QB)) * QB
    last, K2 = (QC, QB) if QC > 1 else (QB, 1)
    out = {}
    for q in range(QA * K2):
        k2, k1 = divmod(q, QA)
        for col, r in enumerate(residues):
            t0 = r + R * q
            assert t0 < M
            at = (QC * k2 * QAP + k1) * P + col + QAP * P * np.arange(last)
            v = np.fft.ifft(tile[at] * w(M, t0) ** np.arange(last)) * last
            for m in range(last):
                out[t0 + R * QA * K2 * m] = v[m]
    return out


@pytest.mark.parametrize("QA,QB,QC,P,M,fold", [
    (4, 5, 1, 32, 60, 1), (5, 4, 1, 32, 200, 2), (8, 8, 1, 32, 256, 1), (6, 7, 1, 16, 420, 1), (4, 8, 1, 8, 512, 4),
    (4, 4, 5, 4, 240, 1), (5, 6, 4, 2, 480, 3), (8, 4, 8, 4, 1024, 1), (7, 9, 1, 16, 63, 1),
])
def test_columns_equal_the_plain_inverse_dft(QA, QB, QC, P, M, fold):
    rng = np.random.default_rng(QA * 100 + QB * 10 + QC + M)
    N, Q = M * fold, QA * QB * QC
    R = M // Q
    for B, b0 in [(1, 0), (Q, 0), (Q, N - 3), (Q - 1, N - Q // 2), (Q // 2 + 1, 7 % N), (max(1, Q // 3), N - 1),
                  (Q, QB * QC - 1), (Q, 1)]:
        Y = rng.standard_normal(B) + 1j * rng.standard_normal(B)
        k = b0 + np.arange(B)
        ref = np.exp(2j * np.pi * np.outer(np.arange(M), k % M) / M) @ Y
        got = {}
        for r0 in range(0, R, P):
            got.update(zoom_columns(Y, b0, M, N, QA, QB, QC, P, list(range(r0, min(R, r0 + P)))))
        assert sorted(got) == list(range(M))
        np.testing.assert_allclose([got[t] for t in range(M)], ref, rtol=0, atol=1e-11 * np.abs(ref).max())


@pytest.mark.parametrize("QA,QB,QC,M,fold", [(2, 4, 5, 240, 1), (5, 4, 4, 320, 2), (8, 4, 8, 1024, 1), (9, 5, 7, 945, 1)])
def test_two_kernel_form_equals_the_plain_inverse_dft(QA, QB, QC, M, fold):
    """csrc/zoom_wide.cuh: the first kernel's Z[b][t'] and the second's passes."""
    rng = np.random.default_rng(M + QA)
    Qp, N = QB * QC, M * fold
    Q, Rp = QA * Qp, M // Qp
    R = Rp // QA
    for B, b0 in [(1, 0), (Q, N - 2), (Q - 1, N - Q // 2), (Q // 2, 3), (Q, Qp - 1)]:
        Y = rng.standard_normal(B) + 1j * rng.standard_normal(B)
        Z = np.full((Qp, Rp), np.nan, complex)
        for b in range(Qp):
            y, g = np.zeros(QA, complex), np.zeros(QA, int)
            for p in range(QA):
                k = b + Qp * p - b0 % Q
                k += Q + b0 if k < 0 else b0          # the bin of the window [b0, b0 + Q)
                y[p] = Y[k - b0] if k - b0 < B else 0.0
                base = b0 // Qp + (1 if b < b0 % Qp else 0)
                g[p] = (p - base) % QA + base
                assert k == b + Qp * g[p]
            for r in range(R):
                v = np.fft.ifft(y * w(Rp, g * r)) * QA
                Z[b, r + R * np.arange(QA)] = v
        out = np.full(M, np.nan, complex)
        for t1 in range(Rp):
            tile = np.full(Qp, np.nan, complex)
            for b1 in range(QC):
                b2 = np.arange(QB)
                assert QC * t1 < M
                tile[b1 + QC * b2] = np.fft.ifft(Z[b1 + QC * b2, t1] * w(M, QC * t1) ** b2) * QB
            for k2 in range(QB):
                t0 = t1 + Rp * k2
                v = np.fft.ifft(tile[QC * k2 + np.arange(QC)] * w(M, t0) ** np.arange(QC)) * QC
                out[t0 + Rp * QB * np.arange(QC)] = v
        k = b0 + np.arange(B)
        ref = np.exp(2j * np.pi * np.outer(np.arange(M), k % M) / M) @ Y
        np.testing.assert_allclose(out, ref, rtol=0, atol=1e-11 * np.abs(ref).max())
