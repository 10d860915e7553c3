"""Bond lists of small lattices, sites row-major: (number of sites, [(u, v)], [class of each bond])."""


def cluster(lx, ly, j2=False, triangular=False, open_y=False):
    """Square lx x ly, periodic; j2: both diagonals (class 1); triangular: one diagonal (class 0)."""
    bonds, cls = [], []
    for y in range(ly):
        for x in range(lx):
            steps = [(1, 0, 0), (0, 1, 0)] + ([(1, 1, 0)] if triangular else []) + ([(1, 1, 1), (-1, 1, 1)] if j2 else [])
            for dx, dy, c in steps:
                if open_y and y + dy >= ly:
                    continue
                bonds.append((x + lx * y, (x + dx) % lx + lx * ((y + dy) % ly)))
                cls.append(c)
    return lx * ly, bonds, cls


def ring(n, *distances):
    return (n, [(i, (i + d) % n) for d in distances for i in range(n)],
            [k for k in range(len(distances)) for _ in range(n)])


# name: (lattice, the split K that holds it with one class for each kind of bond, if any does)
LATTICES = {
    "triangular 4x4": (cluster(4, 4, triangular=True), 12),
    "square 6x3": (cluster(6, 3), 12),
    "square 7x3": (cluster(7, 3), 14),
    "ladder 8x2": (cluster(8, 2, j2=True, open_y=True), 12),
    "ladder 10x2": (cluster(10, 2, j2=True, open_y=True), 15),
    "triangular 4x3": (cluster(4, 3, triangular=True), 10),
    "J1-J2 square 4x3": (cluster(4, 3, j2=True), 10),
    "J1-J2 square 3x4": (cluster(3, 4, j2=True), 10),
    "ring 13, J1 J5": (ring(13, 1, 5), 9),
    "ring 15, J1 J7": (ring(15, 1, 7), 11),
    "ring 18, J1 J2": (ring(18, 1, 2), 11),
    "square 4x4": (cluster(4, 4), 10),
    "square 6x4": (cluster(6, 4), 14),
    # two sites wide: the bonds along y come twice
    "square 6x2 torus": (cluster(6, 2), 9),
    "square 8x2 torus": (cluster(8, 2), 12),
    "triangular 6x2 torus": (cluster(6, 2, triangular=True), None),
}
