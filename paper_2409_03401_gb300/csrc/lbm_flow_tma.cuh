// The fused two-buffer flow step of large FP32 D3Q7 lattices, its loads staged by TMA.
//
// As in fused_flow_kernel a block marches along z and forms phi of plane z + 1 before it
// collides plane z; here one block of 480 threads owns a 32 x 15 tile and the whole SM, and
// every population it reads arrives in shared memory by tensor copies: the scalar sets of a
// plane with a one-node halo, at their pull sources, in a ring of three planes (the plane
// collided, the plane whose phi is formed, the plane in flight), and the flow populations of
// one plane. The gathers of the other kernel keep a warp waiting twice a plane and hold its
// registers meanwhile; here 100 KB are in flight whatever the warps do, no load instruction or
// address is left per population, and nothing is parked. 512^3, a step: 8.19 -> 7.39 ms (0.77 ->
// 0.86 of the copy bandwidth at 320 B a node); tiles inside the lattice alone run at 0.94, bound
// by HBM (with every copy left out the rest takes 4.6 ms); the tiles at the lattice's ends, which
// the copies do not wrap around, take 1.4 times as long at an end in x, hardly longer in y.
#pragma once

#include <cuda.h>

namespace lbm {

namespace tma {

constexpr int X = 32, Y = 15, T = X * Y, Halo = 2 * (X + 2) + 2 * Y;
constexpr int Warps = T / 32;
using L7 = Scalar<LAT_D3Q7>;

// Box of scalar population k: rows y0 - 1 - e_y .. (17 of them), columns from x0 - 4 (e_x = 0:
// 40, e_x = 1: 36) or x0 (e_x = -1: 36), so that a row starts on 16 bytes. Ring position (i, j),
// node (x0 - 1 + j, y0 - 1 + i), finds its population at row i, column j + col.
__host__ __device__ constexpr int s_pitch(int k) { return L7::ex(k) == 0 ? 40 : 36; }
__host__ __device__ constexpr int s_col(int k) { return L7::ex(k) == 0 ? 3 : (L7::ex(k) > 0 ? 2 : 0); }
__host__ __device__ constexpr int s_start(int k) { return L7::ex(k) < 0 ? 0 : -4; }
__host__ __device__ constexpr int s_bytes(int k) { return s_pitch(k) * (Y + 2) * 4; }
__host__ __device__ constexpr int s_room(int k) { return (s_bytes(k) + 127) / 128 * 128; }
__host__ __device__ constexpr int s_off(int set, int k) {              // k = 1, 2 are the populations along x
    const int wide = s_room(0), narrow = s_room(1), along_x = k > 2 ? 2 : (k > 0 ? k - 1 : 0);
    return set * (5 * wide + 2 * narrow) + (k - along_x) * wide + along_x * narrow;
}
constexpr int kPlaneRoom = s_off(3, 0);
// Box of flow population k: rows y0 - e_y .. (15), columns from x0 (e_x = 0: 32, e_x = -1: 36) or
// x0 - 4 (e_x = 1: 36).
__host__ __device__ constexpr int f_pitch(int k) { return D3Q19::ex(k) == 0 ? 32 : 36; }
__host__ __device__ constexpr int f_col(int k) { return D3Q19::ex(k) == 0 ? 0 : (D3Q19::ex(k) > 0 ? 3 : 1); }
__host__ __device__ constexpr int f_start(int k) { return D3Q19::ex(k) > 0 ? -4 : 0; }
__host__ __device__ constexpr int f_bytes(int k) { return f_pitch(k) * Y * 4; }
__host__ __device__ constexpr int f_room(int k) { return (f_bytes(k) + 127) / 128 * 128; }
__host__ __device__ constexpr int f_off(int k) {                       // one bit per k with e_x != 0
    int shifted = 0;
    for (unsigned m = 0x1E786u & ((1u << k) - 1u); m; m &= m - 1u) ++shifted;
    return (k - shifted) * f_room(0) + shifted * f_room(1);
}
__host__ __device__ constexpr bool boxes_are_packed() {
    for (int k = 0; k < 19; ++k)
        if (f_off(k + 1) - f_off(k) != f_room(k)) return false;
    for (int k = 0; k < 7; ++k)
        if (s_off(0, k + 1) - s_off(0, k) != s_room(k)) return false;
    return s_off(1, 0) == s_off(0, 7);
}
static_assert(boxes_are_packed(), "rooms of the boxes in shared memory");
constexpr int kFlowRoom = f_off(19);
constexpr int kRing = 4 * (Y + 2) * (X + 2) * 4;
// Values that come in over the lattice's end, for the tiles there: each thread's own, by cp.async.
struct Ends {
    float f_x[5][Y], f_y[5][X];                        // flow populations of the plane collided next
    float s_x[3][3][Y], s_y[3][3][X];                  // scalar populations along x and y, three planes
};
constexpr int kSmem = 3 * kPlaneRoom + kFlowRoom + kRing + 64 + int(sizeof(Ends));
static_assert(kPlaneRoom % 128 == 0 && kFlowRoom % 128 == 0 && kSmem <= 232448, "shared memory of one SM");

// Components of the velocities plus one, two bits each.
template <class L>
__host__ __device__ constexpr unsigned long long packed(int axis) {
    unsigned long long p = 0;
    for (int k = 0; k < L::Q; ++k)
        p |= (unsigned long long)((axis == 0 ? L::ex(k) : (axis == 1 ? L::ey(k) : L::ez(k))) + 1) << (2 * k);
    return p;
}
constexpr unsigned long long kEx7 = packed<L7>(0), kEy7 = packed<L7>(1), kEz7 = packed<L7>(2);
constexpr unsigned long long kEx19 = packed<D3Q19>(0), kEy19 = packed<D3Q19>(1), kEz19 = packed<D3Q19>(2);

// the tensor maps of a state copy: x, y, z and the 40 planes, in boxes of the four shapes
struct Maps { CUtensorMap s0, s1, f0, f1; };

__device__ __forceinline__ unsigned addr(const void* p) { return unsigned(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void bar_init(unsigned b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned b, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
}
// Waits for a phase of a barrier; false after a bounded number of tries.
__device__ __forceinline__ bool bar_wait(unsigned b, unsigned parity) {
    for (int i = 0; i < (1 << 20); ++i) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(b), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void fetch(float& to, const float* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(addr(&to)), "l"(from) : "memory");
}
__device__ __forceinline__ void load_box(unsigned to, const CUtensorMap* m, int x, int y, int z, int plane, unsigned b) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(to), "l"(m), "r"(x), "r"(y), "r"(z), "r"(plane), "r"(b) : "memory");
}

}  // namespace tma

template <int COLL>
__global__ void __launch_bounds__(tma::T, 1)
flow_tma_kernel(const DevParams P, const __grid_constant__ tma::Maps maps, const StateView src, const StateView dst,
                const float* rim_phi, unsigned* fault, int zchunk) {
    using namespace tma;
    constexpr int kColl = COLL == 2 ? 2 : -1;
    extern __shared__ __align__(128) unsigned char tma_smem[];
    unsigned char* flow = tma_smem + 3 * kPlaneRoom;
    float (*ring)[Y + 2][X + 2] = reinterpret_cast<float (*)[Y + 2][X + 2]>(flow + kFlowRoom);
    const unsigned bars = addr(flow + kFlowRoom + kRing);              // three scalar planes, the flow plane
    Ends& ends = *reinterpret_cast<Ends*>(flow + kFlowRoom + kRing + 64);
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    // the last tile of a row (column) ends with the lattice and leaves what the one before owns
    const int x0 = min(int(blockIdx.x) * X, P.nx - X), y0 = min(int(blockIdx.y) * Y, P.ny - Y);
    const int zs = blockIdx.z * zchunk, ze = min(zs + zchunk, P.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x >= int(blockIdx.x) * X && y >= int(blockIdx.y) * Y;
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) bar_init(bars + 8 * i, Warps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    begin_after_previous();
    __syncthreads();

    // lattice plane whose phi stands for plane zz: periodic, or mirrored across a z wall
    auto plane_of = [&](int zz) {
        if (zz < 0) return P.wall_z ? 0 : zz + P.nz;
        if (zz >= P.nz) return P.wall_z ? P.nz - 1 : zz - P.nz;
        return zz;
    };
    // source of a population moving along ez into plane z: plane, and whether it bounced at a wall
    auto z_source = [&](int z, int ez, bool& bounced) {
        const int q = z - ez;
        bounced = P.wall_z && (q < 0 || q >= P.nz);
        return bounced ? z : (q < 0 ? q + P.nz : (q >= P.nz ? q - P.nz : q));
    };
    // Every warp's first lane issues its share of the boxes of a plane: scalar populations (sets in
    // order) ty and ty + 15 of 21, flow populations ty and ty + 15 of 19. One box's code in a loop,
    // not forty: a plane's pass over the code is long for the instruction cache as it is.
    auto component = [](unsigned long long packed, int k) { return int(packed >> (2 * k) & 3ull) - 1; };
    auto load_scalars = [&](int zz, int slot) {
        if (tx != 0) return;
        const int z = plane_of(zz);
        const unsigned b = bars + 8 * slot, to = addr(tma_smem) + slot * kPlaneRoom;
        bar_expect(b, s_bytes(ty % 7) + (ty + Warps < 21 ? s_bytes((ty + Warps) % 7) : 0));
#pragma unroll 1
        for (int i = ty; i < 21; i += Warps) {
            const int set = i / 7, k = i - 7 * set;
            const int ex = component(kEx7, k), ey = component(kEy7, k), ez = component(kEz7, k);
            bool bounced;
            const int zq = z_source(z, ez, bounced);
            load_box(to + s_off(set, k), ex == 0 ? &maps.s0 : &maps.s1, x0 + s_start(k), y0 - 1 - ey, zq,
                     19 + i + (bounced ? opp(k) - k : 0), b);
        }
    };
    auto load_flow = [&](int z) {
        if (tx != 0) return;
        const unsigned b = bars + 24, to = addr(flow);
        bar_expect(b, f_bytes(ty) + (ty + Warps < 19 ? f_bytes(ty + Warps) : 0));
#pragma unroll 1
        for (int k = ty; k < 19; k += Warps) {
            const int ex = component(kEx19, k), ey = component(kEy19, k), ez = component(kEz19, k);
            bool bounced;
            const int zq = z_source(z, ez, bounced);
            load_box(to + f_off(k), ex == 0 ? &maps.f0 : &maps.f1, x0 + f_start(k), y0 - ey, zq, k, b);
        }
    };

    // scalar populations of ring position (i, j) of the plane in ``slot``
    auto scalars_at = [&](int slot, int i, int j, Node<float, LAT_D3Q7, false>& nd) {
        const unsigned char* p = tma_smem + slot * kPlaneRoom;
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const int e = (i * s_pitch(k) + j + s_col(k)) * 4;
            nd.g[k] = *reinterpret_cast<const float*>(p + s_off(0, k) + e);
            nd.hA[k] = *reinterpret_cast<const float*>(p + s_off(1, k) + e);
            nd.hB[k] = *reinterpret_cast<const float*>(p + s_off(2, k) + e);
        }
    };
    int hi = 0, hj = 0;
    if (tid < Halo) {
        if (tid < X + 2) { hi = 0; hj = tid; }
        else if (tid < 2 * (X + 2)) { hi = Y + 1; hj = tid - (X + 2); }
        else if (tid < 2 * (X + 2) + Y) { hi = tid - 2 * (X + 2) + 1; hj = 0; }
        else { hi = tid - 2 * (X + 2) - Y + 1; hj = X + 1; }
    }
    const int hx = x0 - 1 + hj, hy = y0 - 1 + hi;

    // ``ok``: every copy so far arrived, for the whole block from the next __syncthreads_and on.
    bool ok = true;
    auto wait = [&](unsigned b, unsigned parity) { if (ok) ok = bar_wait(b, parity & 1); };
    auto scalars_phase = [&](int zz) { return unsigned(zz - (zs - 1)) / 3; };
    auto wait_scalars = [&](int zz, int slot) { wait(bars + 8 * slot, scalars_phase(zz)); };
    // A wait ran out before plane z was collided: no more copies, those in flight (scalars up to
    // plane ``last``, the flow of plane z) land or are waited for once more, before the block's
    // shared memory goes to another; the fault word is set, and the planes the block has not
    // written are marked as not finite.
    auto give_up = [&](int z, int last) {
        for (int zz = max(last - 2, zs - 1); zz <= last; ++zz)
            bar_wait(bars + 8 * ((zz - (zs - 1)) % 3), scalars_phase(zz) & 1);
        bar_wait(bars + 24, unsigned(z - zs) & 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (tid == 0) *fault = kWaitFault;
        if (active)
            for (int zz = z; zz < ze; ++zz)
                static_cast<float*>(dst.plane[Planes<LAT_D3Q7>::HA])[node_of(x, y, zz, P)] = __int_as_float(0x7fc00000);
    };

    // Tiles whose sources reach past the lattice's end in x or y, where the copies leave zeros: the
    // threads fetch the wrapped values themselves, most of a plane's time ahead like the copies (a
    // load at the time of use waits behind those in flight, and cost such a tile 3.7 times the
    // plane's time). An end node takes the scalars that come in over the end, three planes deep,
    // and its flow populations that do; a halo thread beside an end takes its node's phi from a
    // field that rim_phi_kernel filled (its 21 scalars cost such a tile another 40 %).
    const bool edge = x0 < 2 || x0 + X + 2 > P.nx || y0 < 2 || y0 + Y + 2 > P.ny;
    const bool ex_p = x == 0, ex_m = x == P.nx - 1;                    // e_x > 0 (< 0) comes over the end
    const bool ey_p = y == 0, ey_m = y == P.ny - 1;
    const bool h_end = edge && tid < Halo && (hx < 1 || hx > P.nx - 2 || hy < 1 || hy > P.ny - 2);
    const int nxy = P.nx * P.ny;
    auto plane_at = [&](int k) { return static_cast<const float*>(src.plane[k]); };
    auto wrap_x = [&](int q) { return q < 0 ? q + P.nx : (q >= P.nx ? q - P.nx : q); };
    auto wrap_y = [&](int q) { return q < 0 ? q + P.ny : (q >= P.ny ? q - P.ny : q); };
    auto fetch_scalars = [&](int zz) {
        const int z = plane_of(zz) * nxy, slot = (zz + 3) % 3;
        if (ex_p || ex_m) {
            const int n = z + y * P.nx + (ex_p ? P.nx - 1 : 0), k = 19 + (ex_p ? 1 : 2);
#pragma unroll
            for (int s = 0; s < 3; ++s) fetch(ends.s_x[slot][s][ty], plane_at(k + 7 * s) + n);
        }
        if (ey_p || ey_m) {
            const int n = z + (ey_p ? P.ny - 1 : 0) * P.nx + x, k = 19 + (ey_p ? 3 : 4);
#pragma unroll
            for (int s = 0; s < 3; ++s) fetch(ends.s_y[slot][s][tx], plane_at(k + 7 * s) + n);
        }
    };
    auto fetch_flow = [&](int z) {
        bool bounced;
        const int zb[3] = {z_source(z, -1, bounced) * nxy, z * nxy, z_source(z, 1, bounced) * nxy};
        if (ex_p || ex_m) {
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                constexpr int kp[5] = {1, 7, 9, 13, 15}, km[5] = {2, 8, 10, 14, 16};
                const int k = ex_p ? kp[i] : km[i];
                const int ey = ex_p ? D3Q19::ey(kp[i]) : D3Q19::ey(km[i]), ez = ex_p ? D3Q19::ez(kp[i]) : D3Q19::ez(km[i]);
                fetch(ends.f_x[i][ty], plane_at(k) + zb[ez + 1] + wrap_y(y - ey) * P.nx + (ex_p ? P.nx - 1 : 0));
            }
        }
        if (ey_p || ey_m) {
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                constexpr int kp[5] = {3, 7, 11, 14, 17}, km[5] = {4, 8, 12, 13, 18};
                const int k = ey_p ? kp[i] : km[i];
                const int ex = ey_p ? D3Q19::ex(kp[i]) : D3Q19::ex(km[i]), ez = ey_p ? D3Q19::ez(kp[i]) : D3Q19::ez(km[i]);
                fetch(ends.f_y[i][tx], plane_at(k) + zb[ez + 1] + (ey_p ? P.ny - 1 : 0) * P.nx + wrap_x(x - ex));
            }
        }
    };
    // phi of a halo node beside an end, from rim_phi_kernel
    float h_phi = 0.f, h_next = 0.f;
    const float* h_at = rim_phi + (h_end ? wrap_y(hy) * P.nx + wrap_x(hx) : 0);
    auto fetch_halo = [&](int zz) {
        if (h_end) h_next = h_at[(long long)plane_of(zz) * nxy];
    };
    auto fetched = [] { asm volatile("cp.async.wait_all;" ::: "memory"); };   // this thread's own

    // this thread's scalars of plane zz in ``slot``, and their moments
    auto own_scalars = [&](int zz, int slot, Node<float, LAT_D3Q7, false>& nd) {
        scalars_at(slot, ty + 1, tx + 1, nd);
        if (edge) {
            const int e = (zz + 3) % 3;
            const float (*a)[Y] = ends.s_x[e];
            const float (*b)[X] = ends.s_y[e];
            if (ex_p) { nd.g[1] = a[0][ty]; nd.hA[1] = a[1][ty]; nd.hB[1] = a[2][ty]; }
            if (ex_m) { nd.g[2] = a[0][ty]; nd.hA[2] = a[1][ty]; nd.hB[2] = a[2][ty]; }
            if (ey_p) { nd.g[3] = b[0][tx]; nd.hA[3] = b[1][tx]; nd.hB[3] = b[2][tx]; }
            if (ey_m) { nd.g[4] = b[0][tx]; nd.hA[4] = b[1][tx]; nd.hB[4] = b[2][tx]; }
        }
        nd.moments(P);
    };
    auto fill_own = [&](int zz, int slot) {
        Node<float, LAT_D3Q7, false> nd;
        own_scalars(zz, slot, nd);
        ring[zz & 3][ty + 1][tx + 1] = nd.phi();
    };
    auto fill_halo = [&](int zz, int slot) {
        if (tid < Halo) {
            float v = h_phi;
            if (!h_end) {
                Node<float, LAT_D3Q7, false> nd;
                scalars_at(slot, hi, hj, nd);
                nd.moments(P);
                v = nd.phi();
            }
            ring[zz & 3][hi][hj] = v;
        }
    };

    load_scalars(zs - 1, 0);
    load_scalars(zs, 1);
    load_flow(zs);
    load_scalars(zs + 1, 2);
    if (edge) {
        fetch_scalars(zs - 1);
        fetch_scalars(zs);
        fetch_scalars(zs + 1);
        fetch_halo(zs - 1);
        h_phi = h_next;
        fetch_halo(zs);
        fetched();
    }
    wait_scalars(zs - 1, 0);
    fill_own(zs - 1, 0);
    fill_halo(zs - 1, 0);
    ok = __syncthreads_and(ok);                                        // slot 0 is free again
    if (!ok) return give_up(zs, zs + 1);
    if (zs + 1 < ze) load_scalars(zs + 2, 0);
    if (edge) {
        if (zs + 1 < ze) fetch_scalars(zs + 2);
        fetch_flow(zs);
        h_phi = h_next;
        fetch_halo(zs + 1);
    }
    wait_scalars(zs, 1);
    fill_own(zs, 1);
    fill_halo(zs, 1);
    int slot = 1;                                                      // of plane z
    for (int z = zs; z < ze; ++z) {
        const int next = slot == 2 ? 0 : slot + 1;
        wait_scalars(z + 1, next);
        fill_own(z + 1, next);
        Node<float, LAT_D3Q7, true> nd;
        {
            Node<float, LAT_D3Q7, false> own;
            own_scalars(z, slot, own);
#pragma unroll
            for (int k = 0; k < 7; ++k) { nd.g[k] = own.g[k]; nd.hA[k] = own.hA[k]; nd.hB[k] = own.hB[k]; }
            nd.S = own.S; nd.dcA = own.dcA; nd.dcB = own.dcB;
        }
        h_phi = h_next;
        fill_halo(z + 1, next);
        wait(bars + 24, unsigned(z - zs));                             // the copy issued last
#pragma unroll
        for (int k = 0; k < 19; ++k)
            nd.f[k] = *reinterpret_cast<const float*>(flow + f_off(k) + (ty * f_pitch(k) + tx + f_col(k)) * 4);
        if (edge) {
            fetched();
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                constexpr int xp[5] = {1, 7, 9, 13, 15}, xm[5] = {2, 8, 10, 14, 16};
                constexpr int yp[5] = {3, 7, 11, 14, 17}, ym[5] = {4, 8, 12, 13, 18};
                if (ex_p) nd.f[xp[i]] = ends.f_x[i][ty];
                if (ex_m) nd.f[xm[i]] = ends.f_x[i][ty];
                if (ey_p) nd.f[yp[i]] = ends.f_y[i][tx];
                if (ey_m) nd.f[ym[i]] = ends.f_y[i][tx];
            }
        }
        // phi of plane z + 1 is there; slot and flow are read no more
        ok = __syncthreads_and(ok);
        if (!ok) return give_up(z, z + 1 < ze ? z + 2 : z + 1);
        // the flow first: it is wanted in a plane's time, the scalars in two (8.6 ms a step at 512^3
        // the other way round)
        if (z + 1 < ze) load_flow(z + 1);
        if (edge && z + 1 < ze) {
            fetch_flow(z + 1);
            fetch_halo(z + 2);
            if (z + 2 < ze) fetch_scalars(z + 3);
        }
        if (z + 2 < ze) load_scalars(z + 3, slot);
        if (active) {
            const int self = node_of(x, y, z, P);
            if (P.wall_z && (z == 0 || z == P.nz - 1)) {               // bounced at the wall: the node's own
#pragma unroll
                for (int k = 1; k < 19; ++k)
                    if ((D3Q19::ez(k) > 0 && z == 0) || (D3Q19::ez(k) < 0 && z == P.nz - 1))
                        nd.f[k] = static_cast<const float*>(src.plane[opp(k)])[self];
            }
            const int sp = (z - 1) & 3, sc = z & 3, sn = (z + 1) & 3;
            const float phi = ring[sc][ty + 1][tx + 1];
            float gx, gy, gz, lap, Fx, Fy, Fz, ux, uy, uz;
            stencil([&](int dx, int dy, int dz) {
                        return ring[dz < 0 ? sp : (dz > 0 ? sn : sc)][ty + 1 + dy][tx + 1 + dx];
                    }, phi, gx, gy, gz, lap);
            force_velocity(nd, phi, gx, gy, gz, lap, P, Fx, Fy, Fz, ux, uy, uz);
            collide_store<float, LAT_D3Q7, true, AddrInterior, kColl>(nd, phi, ux, uy, uz, Fx, Fy, Fz, dst,
                                                                      AddrInterior{self, P.nx, P.nx * P.ny}, P);
        }
        slot = next;
    }
}

// phi of the nodes at the ends of the lattice in x and y, which tiles at the opposite ends read.
static __global__ void __launch_bounds__(kBlockX)
rim_phi_kernel(const DevParams P, const StateView st, float* phi_out) {
    begin_after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, z = blockIdx.z;
    const int rows = 2 * P.nx, c = i - rows;
    if (i >= rows + 2 * (P.ny - 2)) return;
    const int x = i < rows ? (i < P.nx ? i : i - P.nx) : (c < P.ny - 2 ? 0 : P.nx - 1);
    const int y = i < rows ? (i < P.nx ? 0 : P.ny - 1) : 1 + (c < P.ny - 2 ? c : c - (P.ny - 2));
    Addr<PULL> ad;
    ad.self = node_of(x, y, z, P);
    ad.nb.init(x, y, z, P);
    Node<float, LAT_D3Q7, false> nd;
    nd.gather_scalars(st, ad, P);
    nd.moments(P);
    phi_out[ad.self] = nd.phi();
}

// Tensor maps of a state copy; false where the driver refuses them.
inline bool tma_maps(const DevParams& P, const StateView& st, tma::Maps& m) {
    using Encode = decltype(&cuTensorMapEncodeTiled);
    static const Encode encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &r) != cudaSuccess ||
            r != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<Encode>(fn);
    }();
    if (!encode) return false;
    const cuuint64_t dim[4] = {cuuint64_t(P.nx), cuuint64_t(P.ny), cuuint64_t(P.nz), 40};
    const cuuint64_t stride[3] = {cuuint64_t(P.nx) * 4, cuuint64_t(P.nx) * P.ny * 4, cuuint64_t(P.plane) * 4};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    auto make = [&](CUtensorMap& out, int w, int h) {
        const cuuint32_t box[4] = {cuuint32_t(w), cuuint32_t(h), 1, 1};
        return encode(&out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, st.f, dim, stride, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    return make(m.s0, 40, tma::Y + 2) && make(m.s1, 36, tma::Y + 2) && make(m.f0, 32, tma::Y) && make(m.f1, 36, tma::Y);
}

}  // namespace lbm
