// Emitter of the tile kernel of the net production rates (32 states per block, all
// exponents in fixed point): the mechanism's tables and sizes for pyro_tile.cuh.
#pragma once

#include <string>

#include "pyro_emit.h"
#include "pyro_mech.h"

namespace pyro {

struct TileEmit {
  std::string source;      // empty: the mechanism does not fit the tables (see why)
  std::string why;
  int warps = 8;           // per block
  int smem_bytes = 0;      // dynamic shared memory per block
  double t_lo = 0.0;       // states at or below it are left to the FP64 kernel
  int chunks = 0, rows = 0;
  int scratch_bytes = 0;   // global scratch per block (dense Jacobian)
};

// Dynamic shared memory an SM can hold, and what a resident block costs beside its own.
constexpr int kSmemPerSm = 228 * 1024;
constexpr int kSmemPerBlock = 1024;
constexpr int kSmemMaxBlock = 227 * 1024;

// Kernels over the tables: net production rates (pyro_tile.cuh), Jacobian-vector product
// (pyro_tile_jvp.cuh), vector-Jacobian product (pyro_tile_vjp.cuh), dense Jacobian
// (pyro_tile_jac.cuh).
enum class TileKind { Rates, Jvp, Vjp, Jac };
TileEmit emit_tile_unit(const Mechanism& m, TileKind kind = TileKind::Rates);

struct TransportTile {
  std::string source;      // empty: no transport section, or its fits do not suit the tables
  int warps = 0, smem_bytes = 0;
};

TransportTile emit_transport_tile(const Mechanism& m);

// The kernel texts (embedded at build time).
extern const char* kFixedMathSource;
extern const char* kTileSource;
extern const char* kTransportSource;
extern const char* kTileJvpSource;
extern const char* kTileVjpSource;
extern const char* kTileJacSource;

}  // namespace pyro
