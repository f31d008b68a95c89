"""How the rotate + quantize team kernel cuts its CTA (host arithmetic only)."""
import ctypes as C

import pytest


class TeamShape(C.Structure):
    _fields_ = [("R", C.c_int), ("team_warps", C.c_int), ("teams", C.c_int), ("smem", C.c_size_t), ("use", C.c_double)]


def _shape(M, K, asym):
    from paper_2503_06564_b200 import trdq
    f = getattr(trdq.lib(), "_ZN4trdq26rotate_quantize_team_shapeEiiibPNS_9TeamShapeE")
    f.restype, f.argtypes = C.c_bool, [C.c_int, C.c_int, C.c_int, C.c_bool, C.POINTER(TeamShape)]
    s = TeamShape()
    return s if f(M, K, 148, asym, C.byref(s)) else None


@pytest.mark.parametrize("asym", [False, True])
def test_shapes_fit(asym):
    for K in range(128, 18432, 128):
        for M in (148, 1 << 20):
            s = _shape(M, K, asym)
            if s:
                assert s.teams >= 2 and s.teams * s.team_warps <= 12 and 1 <= s.R <= 32 and s.R * (K // 128) <= 32 * s.team_warps
                # two input stages and a code tile per team, the fused vector, the row-exchange table(s), two barriers per team
                table = s.teams * 3 * s.R * 4 * (2 if asym else 1)
                assert s.smem <= 227 * 1024 and s.smem >= s.teams * 5 * s.R * K + K // 128 * 132 * 4 + table + s.teams * 16


def test_the_symmetric_form_does_not_pay_for_the_asymmetric_tables():
    assert (_shape(1 << 20, 128, False).teams, _shape(1 << 20, 128, True).teams) == (11, 10)
    for K in range(256, 18432, 128):
        a, b = _shape(1 << 20, K, False), _shape(1 << 20, K, True)
        assert (a is None) == (b is None) and (a is None or (a.R, a.team_warps, a.teams) == (b.R, b.team_warps, b.teams))
