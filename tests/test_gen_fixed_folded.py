"""The generated fixed-point evaluation of mechanisms with a large fuel.  The species
that element conservation eliminates (CO2, H2O, O2) enter the kept species' enthalpies
with coefficients up to the fuel's atom counts: h/RT of the combination is the fuel's
heat of combustion, 1800 for n-heptane and 2800 for n-undecane at 300 K, beyond
what 53 fraction bits leave of a 64-bit word.  Compared with the FP64 evaluation by the host build
of test_gen_fixed_host."""
import pytest

import test_gen_fixed_host as host

# name: atoms C H O N, heat of formation [kJ/mol], S/R at 298 K, cp/R = a1 + a2 T
_BASE = {"H2": ((0, 2, 0, 0), 0.0, 15.7, 3.3, 4e-4), "O2": ((0, 0, 2, 0), 0.0, 24.7, 3.5, 4e-4),
         "H": ((0, 1, 0, 0), 218.0, 13.8, 2.5, 0.0), "O": ((0, 0, 1, 0), 249.2, 19.4, 2.5, 0.0),
         "OH": ((0, 1, 1, 0), 37.3, 22.1, 3.5, 3e-4), "HO2": ((0, 1, 2, 0), 12.0, 27.6, 4.5, 1e-3),
         "H2O": ((0, 2, 1, 0), -241.8, 22.7, 4.0, 1e-3), "CO": ((1, 0, 1, 0), -110.5, 23.8, 3.5, 4e-4),
         "CO2": ((1, 0, 2, 0), -393.5, 25.7, 5.0, 1e-3), "CH3": ((1, 3, 0, 0), 146.7, 23.4, 5.0, 2e-3),
         "CH2O": ((1, 2, 1, 0), -108.6, 26.3, 5.0, 2e-3), "C2H4": ((2, 4, 0, 0), 52.4, 26.4, 6.0, 4e-3),
         "C3H7": ((3, 7, 0, 0), 100.5, 34.8, 10.0, 8e-3)}
# (some lumped to three entries a side; CO2, H2O and O2 take part most)
_RX = [("H O2", "OH O", 1e14, 0.0, 70.0), ("O H2", "OH H", 5e4, 2.7, 26.0), ("OH H2", "H2O H", 2e8, 1.5, 14.0),
       ("OH OH", "H2O O", 3e4, 2.4, 0.0), ("CO OH", "CO2 H", 5e7, 1.3, 3.0), ("CO HO2", "CO2 OH", 1e13, 0.0, 90.0),
       ("CO O2", "CO2 O", 2e12, 0.0, 200.0), ("CO H2O", "CO2 H2", 1e9, 1.0, 150.0), ("CO O", "CO2", 6e10, 0.0, 10.0),
       ("CH2O O2", "CO2 H2O", 1e12, 0.0, 160.0), ("CH2O O", "CO2 H2", 1e12, 0.0, 20.0), ("CH2O OH", "CO H2O H", 3e13, 0.0, 5.0),
       ("CH3 O", "CH2O H", 8e13, 0.0, 0.0), ("C2H4 O2", "CH2O CH2O", 1e12, 0.0, 120.0),
       ("C2H4 OH", "CH3 CH2O", 2e12, 0.0, 4.0), ("HO2 H", "OH OH", 7e13, 0.0, 2.0), ("HO2 OH", "H2O O2", 2e13, 0.0, 0.0),
       ("HO2 H", "H2 O2", 2e13, 0.0, 5.0), ("C3H7", "C2H4 CH3", 1e13, 0.0, 130.0)]


def _alkane(nc):
    """A 16-species skeleton of the oxidation of n-C7H16 or n-C11H24 (lumped to three entries a side)."""
    h = -20.6 * nc - 43.6  # -187.8 kJ/mol for n-heptane
    sp = dict(_BASE)
    fuel, alkyl = f"C{nc}H{2 * nc + 2}", f"C{nc}H{2 * nc + 1}"
    sp[fuel] = ((nc, 2 * nc + 2, 0, 0), h, 7.4 * nc, 3.0 * nc, 4e-3 * nc)
    sp[alkyl] = ((nc, 2 * nc + 1, 0, 0), h + 195.0, 7.4 * nc, 3.0 * nc, 4e-3 * nc)
    rx = list(_RX)
    if nc == 11:
        sp["C7H15"] = ((7, 15, 0, 0), 7.2, 51.5, 21.0, 0.028)
        rx += [(alkyl, "C2H4 C2H4 C7H15", 1e13, 0.0, 260.0), ("C7H15", "C2H4 C2H4 C3H7", 1e13, 0.0, 260.0)]
    else:
        sp["N2"] = ((0, 0, 0, 2), 0.0, 23.0, 3.5, 4e-4)
        rx += [(alkyl, "C2H4 C2H4 C3H7", 1e13, 0.0, 260.0)]
    rx += [(fuel + " OH", alkyl + " H2O", 1e12, 0.0, 5.0), (fuel + " H", alkyl + " H2", 1e13, 0.0, 30.0),
           (fuel + " O2", alkyl + " HO2", 1e13, 0.0, 200.0)]
    species = []
    for k, (c, hf, s, a1, a2) in sp.items():
        species.append({"name": k, "composition": {e: n for e, n in zip("CHON", c) if n}, "T_range": [300.0, 3000.0],
                        "W": sum(w * n for w, n in zip((12.011, 1.008, 15.999, 14.007), c)),
                        "nasa7": [a1, a2, 0.0, 0.0, 0.0, hf * 1e3 / 8.314462618 - 298.15 * (a1 + 0.5 * a2 * 298.15),
                                  s - a1 * 5.6976 - a2 * 298.15]})
    out = []
    for a, b, A, beta, Ea in rx + [("H OH", "H2O", 2e22, -2.0, 0.0), ("H O2", "HO2", 3e19, -1.0, 0.0)]:
        r = {"reactants": {s: a.split().count(s) for s in a.split()}, "products": {s: b.split().count(s) for s in b.split()},
             "type": "elementary", "reversible": True, "A": A, "b": beta, "Ea": Ea, "equation": a + " <=> " + b}
        if A > 1e18:
            r.update(type="three-body", efficiencies={"H2O": 6.0, fuel: 3.0})
        out.append(r)
    assert len(species) == 16
    return {"name": fuel, "elements": ["C", "H", "O", "N"], "units": {"A": "cm, mol, s", "Ea": "kJ/mol", "T": "K"},
            "species": species, "reactions": out}


@pytest.mark.parametrize("nc", [7, 11])
def test_large_fuel(nc, tmp_path, monkeypatch):
    monkeypatch.setitem(host.MECHS, "alkane", lambda: _alkane(nc))
    host.test_fixed_point_evaluation_matches_fp64("alkane", tmp_path)
    src = (tmp_path / "gen.cu").read_text()
    names = [sp["name"] for sp in _alkane(nc)["species"]]
    table = src.split("elim(int e)")[1].split("t[] = {")[1].split("}")[0]
    assert {names[int(k) - 1] for k in table.split(",")[:-1]} == {"CO2", "H2O", "O2"}
